"""Two threads that configure one kernel for different shared-memory sizes at once: the attribute never shrinks (host code,
run on the CPU against stand-ins for the two runtime calls)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include "smem_configured.h"
std::atomic<int> attribute{0};
extern "C" cudaError_t cudaGetDevice(int* dev) { *dev = 0; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int value) {
  if (value == 100) std::this_thread::sleep_for(std::chrono::milliseconds(300));   // the smaller request is the slower one
  attribute = value;
  return cudaSuccess;
}
void kernel() {}
bm::SmemConfigured configured;
int main() {
  std::thread small([] { configured.ensure(kernel, 100); });
  std::this_thread::sleep_for(std::chrono::milliseconds(100));
  std::thread large([] { configured.ensure(kernel, 200); });
  small.join();
  large.join();
  configured.ensure(kernel, 150);
  std::printf("%d\n", attribute.load());
}
"""


def test_shared_memory_attribute_never_shrinks(tmp_path):
    include = "/usr/local/cuda/include"
    if shutil.which("g++") is None or not os.path.isdir(include):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "configured.cpp", tmp_path / "configured"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", include, "-I",
                    os.path.join(ROOT, "paper_2412_05693_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.strip() == "200"
