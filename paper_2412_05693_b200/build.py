"""Builds libbatchmax.so (the C-ABI library) in-tree with nvcc for sm_100a, and the binding's native step where torch is installed.

    python -m paper_2412_05693_b200.build [--force] [--verbose] [--debug]
"""
from __future__ import annotations

import glob
import importlib.metadata
import importlib.util
import os
import subprocess
import sys
import sysconfig

PKG_DIR = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG_DIR, "csrc")
LIB_PATH = os.path.join(PKG_DIR, "libbatchmax.so")
DEBUG_LIB_PATH = os.path.join(PKG_DIR, "libbatchmax_debug.so")   # the checked build: -DBM_DEBUG
FASTCALL_SRC = os.path.join(CSRC, "fastcall.cpp")
HEADER = os.path.join(os.path.dirname(PKG_DIR), "include", "batchmax.h")

NVCC_FLAGS = [
    "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr", "--extended-lambda",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(lib_path: str = LIB_PATH) -> bool:
    if not os.path.exists(lib_path):
        return True
    t = os.path.getmtime(lib_path)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + [HEADER]
    return any(os.path.getmtime(p) > t for p in deps)


def fastcall_path():
    """Where the binding's native step is, or would be, built: it is bound to one torch and one Python (None without torch)."""
    try:
        torch_version = importlib.metadata.version("torch")
    except importlib.metadata.PackageNotFoundError:
        return None
    return os.path.join(PKG_DIR, "_fastcall.torch-" + torch_version.replace("+", "_") + sysconfig.get_config_var("EXT_SUFFIX"))


def build_fastcall(force: bool = False):
    """Compile the binding's native step against torch's headers; returns its path, or None without torch.  The C library needs
    none of it, and the binding goes its general way where it is missing."""
    path, spec = fastcall_path(), importlib.util.find_spec("torch")
    if path is None or spec is None or spec.origin is None:
        return None
    if not force and os.path.exists(path) and os.path.getmtime(path) >= os.path.getmtime(FASTCALL_SRC):
        return path
    torch_dir = os.path.dirname(spec.origin)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [os.path.join(torch_dir, "include"), os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    part = f"{path}.{os.getpid()}"           # (another process may be importing the file, or building it too)
    try:
        subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", *("-I" + d for d in inc), "-o", part, FASTCALL_SRC,
                        "-L" + os.path.join(torch_dir, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"], check=True)
        os.replace(part, path)
    finally:
        if os.path.exists(part):
            os.remove(part)
    return path


def build(force: bool = False, verbose: bool = False, debug: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library; returns its path.  debug: the checked build
    (row-index checks in the kernels, guards behind the slabs), libbatchmax_debug.so."""
    lib_path = DEBUG_LIB_PATH if debug else LIB_PATH
    if not force and not _stale(lib_path):
        return lib_path
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    objs = []
    procs = []
    build_dir = os.path.join(PKG_DIR, "build", "debug" if debug else "release")
    os.makedirs(build_dir, exist_ok=True)
    for src in sources():
        obj = os.path.join(build_dir, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        cmd = [nvcc, *NVCC_FLAGS, *(["-DBM_DEBUG"] if debug else []), "-c", src, "-o", obj]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        procs.append((src, subprocess.Popen(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)))
    failed = False
    for src, p in procs:
        out, _ = p.communicate()
        if p.returncode != 0 or verbose:
            sys.stderr.write(f"--- {os.path.basename(src)}\n{out}\n")
        failed |= p.returncode != 0
    if failed:
        raise RuntimeError("nvcc failed")
    link = [nvcc, "-shared", "-o", lib_path, *objs, "-gencode", "arch=compute_100a,code=sm_100a"]
    subprocess.run(link, check=True)
    return lib_path


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, debug="--debug" in sys.argv))
    build_fastcall(force="--force" in sys.argv)
