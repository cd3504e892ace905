// The two per-step calls of the binding, tsq_encode and tsq_decode on torch tensors, as a CPython extension: argument
// checks, pointers, sizes and the current stream are read from the tensors in C++ and the C ABI (include/tsq.h) is called
// directly.  A decode step is a few microseconds of GPU work, so what the interpreter spends around the call counts: through
// ctypes, with the stream object that torch.cuda.current_stream() builds, a 64 x 4096 decode took 9.1 us of host time per
// call, of which the stream lookup 3.5 us and the argument conversions about 1.5 us.  The interpreter lock is released around the
// call, as ctypes does: a launch can wait for room in the stream's queue.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include "tsq.h"

namespace {

// NULL with a Python error set when `o` is no tensor.
const at::Tensor* tensor(PyObject* o, const char* name) {
  if (!THPVariable_Check(o)) {
    PyErr_Format(PyExc_TypeError, "%s must be a tensor", name);
    return nullptr;
  }
  return &THPVariable_Unpack(o);
}

// None: the current stream of the current device; else an object with a cuda_stream attribute, or the handle as a number.
bool stream_of(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = c10::cuda::getCurrentCUDAStream().stream();
    return true;
  }
  PyObject* handle = PyObject_HasAttrString(o, "cuda_stream") ? PyObject_GetAttrString(o, "cuda_stream") : Py_NewRef(o);
  if (!handle) return false;
  *out = PyLong_AsVoidPtr(handle);
  Py_DECREF(handle);
  return !(*out == nullptr && PyErr_Occurred());
}

// A contiguous [tokens x hidden] CUDA tensor of the plan's type (tokens < 0: any number of rows).
bool check_rows(const at::Tensor& t, long dtype, long hidden, int64_t tokens, const char* name) {
  const at::ScalarType want = dtype == TSQ_BF16 ? at::kBFloat16 : at::kHalf;
  if (t.is_cuda() && t.is_contiguous() && t.scalar_type() == want && t.dim() == 2 && t.size(1) == hidden &&
      (tokens < 0 || t.size(0) == tokens))
    return true;
  PyErr_Format(PyExc_AssertionError, "%s must be a contiguous CUDA tensor [tokens, %ld] of the plan's dtype", name, hidden);
  return false;
}

// encode(plan, dtype, hidden, x, blob, ws, stream) -> status
PyObject* encode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 7) return PyErr_Format(PyExc_TypeError, "encode takes 7 arguments");
  const auto* plan = static_cast<const tsq_plan_t*>(PyLong_AsVoidPtr(a[0]));
  const long dtype = PyLong_AsLong(a[1]), hidden = PyLong_AsLong(a[2]);
  if (PyErr_Occurred()) return nullptr;
  const at::Tensor *x = tensor(a[3], "x"), *blob = x ? tensor(a[4], "blob") : nullptr, *ws = blob ? tensor(a[5], "ws") : nullptr;
  void* stream = nullptr;
  if (!ws || !check_rows(*x, dtype, hidden, -1, "x") || !stream_of(a[6], &stream)) return nullptr;
  const void* xp = x->data_ptr();
  void *bp = blob->data_ptr(), *wp = ws->data_ptr();
  const int64_t tokens = x->size(0);
  const size_t blob_bytes = static_cast<size_t>(blob->numel()), ws_bytes = static_cast<size_t>(ws->numel());
  tsq_status_t st;
  Py_BEGIN_ALLOW_THREADS;
  st = tsq_encode(plan, xp, tokens, bp, blob_bytes, wp, ws_bytes, stream);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

// decode(plan, dtype, hidden, blob, tokens, y, ws, stream) -> status
PyObject* decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  if (n != 8) return PyErr_Format(PyExc_TypeError, "decode takes 8 arguments");
  const auto* plan = static_cast<const tsq_plan_t*>(PyLong_AsVoidPtr(a[0]));
  const long dtype = PyLong_AsLong(a[1]), hidden = PyLong_AsLong(a[2]);
  const long long tokens = PyLong_AsLongLong(a[4]);
  if (PyErr_Occurred()) return nullptr;
  const at::Tensor *blob = tensor(a[3], "blob"), *y = blob ? tensor(a[5], "y") : nullptr, *ws = y ? tensor(a[6], "ws") : nullptr;
  void* stream = nullptr;
  if (!ws || !check_rows(*y, dtype, hidden, tokens, "y") || !stream_of(a[7], &stream)) return nullptr;
  const void* bp = blob->data_ptr();
  void *yp = y->data_ptr(), *wp = ws->data_ptr();
  const size_t blob_bytes = static_cast<size_t>(blob->numel()), ws_bytes = static_cast<size_t>(ws->numel());
  tsq_status_t st;
  Py_BEGIN_ALLOW_THREADS;
  st = tsq_decode(plan, bp, blob_bytes, tokens, yp, wp, ws_bytes, stream);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

// current_stream() -> handle of the current device's current stream
PyObject* current_stream(PyObject*, PyObject*) { return PyLong_FromVoidPtr(c10::cuda::getCurrentCUDAStream().stream()); }

PyMethodDef methods[] = {
    {"encode", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(encode)), METH_FASTCALL, nullptr},
    {"decode", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)(void)>(decode)), METH_FASTCALL, nullptr},
    {"current_stream", current_stream, METH_NOARGS, nullptr},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_tsq_torch", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__tsq_torch(void) { return PyModule_Create(&module); }
