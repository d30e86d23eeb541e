// Argument marshalling of the Python binding, natively: tensors become device pointers, the parameter struct its
// address, the current torch stream the library's stream.  Nothing else happens here; every function
// forwards to the extern "C" entry point of its name and returns its status.
//
// A decode step launches one kernel of 5 to 8 us, and through ctypes a call cost 11 us of host time, five of them
// for fifteen attribute calls and argument conversions in the interpreter: an eager decode loop ran at the
// host's pace.  Measured per calidrop_decode call, host time: 11.2 -> 3.1 us; a
// token of eight layers, called layer by layer: 89 -> 59 us at 4 kv heads x 4333 rows, 89 -> 72 us at 32 x 2111.
#include <Python.h>
#include <c10/cuda/CUDAStream.h>
#include <dlfcn.h>
#include <torch/csrc/autograd/python_variable.h>

#include "../../include/calidrop.h"

namespace {

#define CALIDROP_ENTRIES(X)                                                                                         \
  X(compress) X(calibrate) X(gather_evicted) X(recalibrate) X(accumulated_scores) X(select_from_scores)             \
  X(select_streaming) X(decode) X(decode_batched) X(decode_static)
#define DECLARE(name) decltype(&calidrop_##name) f_##name = nullptr;
CALIDROP_ENTRIES(DECLARE)
#undef DECLARE

// The positional arguments of one call.  A conversion that fails sets a Python error, after which `ok` is
// false and the entry point is not called.
struct Args {
  PyObject* const* a;
  bool ok;
  Args(PyObject* const* args, Py_ssize_t n, Py_ssize_t want) : a(args), ok(n == want) {
    if (!ok) PyErr_Format(PyExc_TypeError, "%zd arguments expected, got %zd", want, n);
  }
  // device pointer of a tensor, a raw address, or null for None
  void* ptr(int i) {
    PyObject* o = a[i];
    if (!ok || o == Py_None) return nullptr;
    if (THPVariable_Check(o)) {
      const at::Tensor& t = THPVariable_Unpack(o);
      if (t.is_contiguous()) return t.data_ptr();
      PyErr_SetString(PyExc_AssertionError, "tensors passed to the library must be contiguous");
      ok = false;
      return nullptr;
    }
    if (PyLong_Check(o)) {
      void* p = PyLong_AsVoidPtr(o);
      ok = !PyErr_Occurred();
      return p;
    }
    PyErr_SetString(PyExc_TypeError, "a tensor, an address or None expected");
    ok = false;
    return nullptr;
  }
  size_t nbytes(int i) {
    if (!ok) return 0;
    if (THPVariable_Check(a[i])) return THPVariable_Unpack(a[i]).nbytes();
    PyErr_SetString(PyExc_TypeError, "the workspace must be a tensor");
    ok = false;
    return 0;
  }
  int32_t i32(int i) {
    if (!ok) return 0;
    PyObject* o = PyLong_Check(a[i]) ? Py_NewRef(a[i]) : PyNumber_Long(a[i]);
    if (!o) { ok = false; return 0; }
    const long v = PyLong_AsLong(o);
    Py_DECREF(o);
    if (v == -1 && PyErr_Occurred()) ok = false;
    else if (v != (int32_t)v) { PyErr_SetString(PyExc_OverflowError, "argument out of the range of int32"); ok = false; }
    return (int32_t)v;
  }
  // address of a ctypes structure or array
  void* buf(int i) {
    if (!ok || a[i] == Py_None) return nullptr;
    Py_buffer v;
    if (PyObject_GetBuffer(a[i], &v, PyBUF_SIMPLE) != 0) { ok = false; return nullptr; }
    void* p = v.buf;
    PyBuffer_Release(&v);   // the caller holds the object for the length of the call
    return p;
  }
  Py_ssize_t len(int i) {
    if (!ok) return 0;
    const Py_ssize_t n = PyObject_Length(a[i]);
    if (n < 0) ok = false;
    return n;
  }
  const calidrop_params* params(int i) { return (const calidrop_params*)buf(i); }
  void* stream() {
    if (!ok) return nullptr;
    try {
      return (void*)c10::cuda::getCurrentCUDAStream().stream();
    } catch (const std::exception& e) {
      PyErr_SetString(PyExc_RuntimeError, e.what());
      ok = false;
      return nullptr;
    }
  }
};

// (the arguments are converted in any order: one that fails turns the later ones into nulls, and no call is made)
template <typename F, typename... A>
PyObject* forward(Args& x, F f, A... v) {
  if (!x.ok) return nullptr;
  int rc;
  Py_BEGIN_ALLOW_THREADS   // a launch may have to wait for room in the stream's queue
  rc = f(v...);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

#define ENTRY(name, n_args, ...)                                                        \
  PyObject* py_##name(PyObject*, PyObject* const* args, Py_ssize_t n) {                 \
    Args x(args, n, n_args);                                                            \
    if (!x.ok) return nullptr;                                                          \
    return forward(x, f_##name, __VA_ARGS__);                                           \
  }

ENTRY(compress, 12, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), (const float*)x.ptr(4), (int32_t*)x.ptr(5), x.ptr(6),
      x.ptr(7), (float*)x.ptr(8), (float*)x.ptr(9), x.ptr(10), x.ptr(11), x.nbytes(11), x.stream())
ENTRY(calibrate, 12, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), (const float*)x.ptr(4), (const int32_t*)x.ptr(5),
      x.ptr(6), x.ptr(7), (float*)x.ptr(8), (float*)x.ptr(9), x.ptr(10), x.ptr(11), x.nbytes(11), x.stream())
ENTRY(gather_evicted, 8, x.params(0), x.ptr(1), x.ptr(2), (const int32_t*)x.ptr(3), (int32_t*)x.ptr(4), x.ptr(5),
      x.ptr(6), x.ptr(7), x.nbytes(7), x.stream())
ENTRY(recalibrate, 10, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), x.i32(4), x.i32(5), (float*)x.ptr(6),
      (float*)x.ptr(7), x.ptr(8), x.ptr(9), x.nbytes(9), x.stream())
ENTRY(accumulated_scores, 5, x.params(0), x.ptr(1), x.ptr(2), (float*)x.ptr(3), x.ptr(4), x.nbytes(4), x.stream())
ENTRY(select_from_scores, 5, x.params(0), (const float*)x.ptr(1), x.i32(2), (int32_t*)x.ptr(3), x.ptr(4), x.nbytes(4),
      x.stream())
ENTRY(select_streaming, 3, x.params(0), x.i32(1), (int32_t*)x.ptr(2), x.stream())
ENTRY(decode, 14, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), x.ptr(4), x.ptr(5), x.i32(6), (const float*)x.ptr(7),
      (const float*)x.ptr(8), x.ptr(9), x.ptr(10), (float*)x.ptr(11), (uint8_t*)x.ptr(12), x.ptr(13), x.nbytes(13),
      x.stream())
ENTRY(decode_batched, 4, x.params(0), (int32_t)x.len(1), (const calidrop_decode_layer*)x.buf(1), x.i32(2), x.ptr(3),
      x.nbytes(3), x.stream())
ENTRY(decode_static, 13, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), x.ptr(4), x.ptr(5), x.i32(6), (const float*)x.ptr(7),
      (const float*)x.ptr(8), x.ptr(9), x.ptr(10), (float*)x.ptr(11), (uint8_t*)x.ptr(12), x.stream())

// open(path): the shared library whose entry points the functions forward to
PyObject* py_open(PyObject*, PyObject* path) {
  const char* s = PyUnicode_AsUTF8(path);
  if (!s) return nullptr;
  void* h = dlopen(s, RTLD_NOW | RTLD_LOCAL);
  if (!h) return PyErr_Format(PyExc_ImportError, "%s", dlerror());
#define RESOLVE(name)                                                                               \
  f_##name = (decltype(f_##name))dlsym(h, "calidrop_" #name);                                        \
  if (!f_##name) return PyErr_Format(PyExc_ImportError, "%s does not export calidrop_" #name, s);
  CALIDROP_ENTRIES(RESOLVE)
#undef RESOLVE
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"open", py_open, METH_O, nullptr},
#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr},
    CALIDROP_ENTRIES(METHOD)
#undef METHOD
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&module); }
