// The two calls that a program makes for every block and every token, from Python tensors to the library's C functions in
// one native step.  A small decode step takes 5 to 7 us on the GPU; checking and marshalling its arguments in Python took
// 3.4 us of the 7.1 us that a step took on the host (the C call with its launch 2.7, ctypes 1.0).
//
// Both functions return the library's status code, or None where an argument is not what they handle (a tensor subclass, a
// stream object, an index that is not an int): binding.py then takes its own, general way.  The checks are that way's
// checks and fail like them, with AssertionError.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

namespace {

typedef int32_t (*DecodeFn)(void*, int32_t, int32_t, int32_t, const void*, const void*, const void*, void*, int32_t, void*);
typedef int32_t (*PrefillFn)(void*, int32_t, int32_t, int32_t, const void*, const void*, const void*, int32_t, int32_t, void*,
                             int32_t, void*);

// int arguments args[0 .. n): false where one is no plain int of 32 bits
bool ints(PyObject* const* args, int n, int32_t* out) {
  for (int i = 0; i < n; ++i) {
    if (!PyLong_CheckExact(args[i])) return false;
    int overflow = 0;
    const long v = PyLong_AsLongAndOverflow(args[i], &overflow);
    if (overflow != 0 || v < INT32_MIN || v > INT32_MAX) return false;
    out[i] = (int32_t)v;
  }
  return true;
}

// q, k, v, out: exact torch.Tensor objects with storage
bool tensors(PyObject* const* args, const at::Tensor** t) {
  for (int i = 0; i < 4; ++i) {
    if (!THPVariable_CheckExact(args[i])) return false;
    t[i] = &THPVariable_Unpack(args[i]);
    if (!t[i]->has_storage()) return false;
  }
  return true;
}

bool layouts_ok(const at::Tensor* const* t, bool bf16) {
  const at::ScalarType want = bf16 ? at::kBFloat16 : at::kFloat;
  if (!t[0]->is_contiguous() || !t[1]->is_contiguous() || !t[2]->is_contiguous() || t[0]->scalar_type() != want) {
    PyErr_SetNone(PyExc_AssertionError);
    return false;
  }
  if (!t[3]->is_contiguous() || t[3]->scalar_type() != want || !t[3]->sizes().equals(t[0]->sizes())) {
    PyErr_SetString(PyExc_AssertionError, "out must be a contiguous tensor of q's shape and dtype");
    return false;
  }
  return true;
}

// (function address, handle, bf16, q, k, v, out, layer, sample0, evict_to)
PyObject* decode(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  int32_t x[3];
  const at::Tensor* t[4];
  if (n != 10 || !tensors(args + 3, t) || !ints(args + 7, 3, x) || t[0]->dim() < 1) Py_RETURN_NONE;
  void* fn = PyLong_AsVoidPtr(args[0]);
  void* h = PyLong_AsVoidPtr(args[1]);
  if (PyErr_Occurred() || !layouts_ok(t, args[2] == Py_True)) return nullptr;
  const void *q = t[0]->data_ptr(), *k = t[1]->data_ptr(), *v = t[2]->data_ptr();
  void* out = t[3]->data_ptr();
  const int32_t ns = (int32_t)t[0]->size(0);
  void* stream = c10::cuda::getCurrentCUDAStream().stream();
  int32_t rc;
  Py_BEGIN_ALLOW_THREADS
  rc = reinterpret_cast<DecodeFn>(fn)(h, x[0], x[1], ns, q, k, v, out, x[2], stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
  END_HANDLE_TH_ERRORS
}

// (function address, handle, bf16, q, k, v, out, layer, sample0, evict_to, pos0)
PyObject* prefill(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  int32_t x[4];
  const at::Tensor* t[4];
  if (n != 11 || !tensors(args + 3, t) || !ints(args + 7, 4, x) || t[0]->dim() < 2) Py_RETURN_NONE;
  void* fn = PyLong_AsVoidPtr(args[0]);
  void* h = PyLong_AsVoidPtr(args[1]);
  if (PyErr_Occurred() || !layouts_ok(t, args[2] == Py_True)) return nullptr;
  const void *q = t[0]->data_ptr(), *k = t[1]->data_ptr(), *v = t[2]->data_ptr();
  void* out = t[3]->data_ptr();
  const int32_t ns = (int32_t)t[0]->size(0), I = (int32_t)t[0]->size(1);
  void* stream = c10::cuda::getCurrentCUDAStream().stream();
  int32_t rc;
  Py_BEGIN_ALLOW_THREADS
  rc = reinterpret_cast<PrefillFn>(fn)(h, x[0], x[1], ns, q, k, v, I, x[3], out, x[2], stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"decode", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(decode)), METH_FASTCALL, nullptr},
    {"prefill", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(prefill)), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__fastcall() { return PyModule_Create(&module); }
