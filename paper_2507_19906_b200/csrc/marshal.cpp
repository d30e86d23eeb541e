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

PyTypeObject* params_type = nullptr;   // the binding's ctypes structures (see open)
PyTypeObject* layer_type = nullptr;

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
    if (PyLong_Check(o)) return address(o);
    if (THPVariable_CheckExact(o)) {
      // (torch throws for a tensor without memory of its own, sparse or wrapped: no exception may leave through
      // the interpreter's frames, and the tensor's own methods raise it properly)
      try {
        const at::Tensor& t = THPVariable_Unpack(o);
        if (t.is_contiguous()) return t.data_ptr();
        not_contiguous();
        return nullptr;
      } catch (...) {
      }
    }
    // subclasses of torch.Tensor and anything else with its methods
    if (!method(o, "data_ptr")) return nullptr;
    PyObject* contiguous = call(o, "is_contiguous");
    if (!contiguous) return nullptr;
    const int c = PyObject_IsTrue(contiguous);
    Py_DECREF(contiguous);
    if (c < 0) ok = false;
    else if (c == 0) not_contiguous();
    if (!ok) return nullptr;
    PyObject* p = call(o, "data_ptr");
    if (!p) return nullptr;
    void* const r = address(p);
    Py_DECREF(p);
    return r;
  }
  size_t nbytes(int i) {
    PyObject* o = a[i];
    if (!ok) return 0;
    if (THPVariable_CheckExact(o)) {
      try {
        return THPVariable_Unpack(o).nbytes();
      } catch (...) {
      }
    }
    if (!method(o, "element_size")) return 0;
    size_t bytes = 1;
    for (const char* m : {"numel", "element_size"}) {
      PyObject* v = call(o, m);
      if (!v) return 0;
      bytes *= PyLong_AsSize_t(v);
      Py_DECREF(v);
      if (PyErr_Occurred()) { ok = false; return 0; }
    }
    return bytes;
  }
  void not_contiguous() {
    PyErr_SetString(PyExc_AssertionError, "tensors passed to the library must be contiguous");
    ok = false;
  }
  void* address(PyObject* o) {
    void* p = PyLong_AsVoidPtr(o);
    if (!p && PyErr_Occurred()) ok = false;
    return p;
  }
  bool method(PyObject* o, const char* name) {
    if (!PyObject_HasAttrString(o, name)) {
      PyErr_SetString(PyExc_TypeError, "a tensor, an address or None expected");
      ok = false;
    }
    return ok;
  }
  PyObject* call(PyObject* o, const char* name) {
    PyObject* r = PyObject_CallMethod(o, name, nullptr);
    if (!r) ok = false;
    return r;
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
  // Structures are taken by their type, as ctypes would: a buffer of other bytes would be read as pointers and sizes.
  const calidrop_params* params(int i) {
    if (!ok) return nullptr;
    if (PyObject_TypeCheck(a[i], params_type)) return (const calidrop_params*)buf(i);
    PyErr_SetString(PyExc_TypeError, "a Params structure expected");
    ok = false;
    return nullptr;
  }
  const calidrop_decode_layer* layers(int i) {
    if (!ok) return nullptr;
    PyObject* element = PyObject_GetAttrString((PyObject*)Py_TYPE(a[i]), "_type_");   // of an array type
    if (!element) PyErr_Clear();
    const bool match = element && element == (PyObject*)layer_type && PyObject_CheckBuffer(a[i]);
    Py_XDECREF(element);
    if (match) return (const calidrop_decode_layer*)buf(i);
    PyErr_SetString(PyExc_TypeError, "an array of DecodeLayer structures expected");
    ok = false;
    return nullptr;
  }
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
  void* const stream = x.stream();
  if (!x.ok) return nullptr;
  int rc;
  Py_BEGIN_ALLOW_THREADS   // a launch may have to wait for room in the stream's queue
  rc = f(v..., stream);
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
      x.ptr(7), (float*)x.ptr(8), (float*)x.ptr(9), x.ptr(10), x.ptr(11), x.nbytes(11))
ENTRY(calibrate, 12, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), (const float*)x.ptr(4), (const int32_t*)x.ptr(5),
      x.ptr(6), x.ptr(7), (float*)x.ptr(8), (float*)x.ptr(9), x.ptr(10), x.ptr(11), x.nbytes(11))
ENTRY(gather_evicted, 8, x.params(0), x.ptr(1), x.ptr(2), (const int32_t*)x.ptr(3), (int32_t*)x.ptr(4), x.ptr(5),
      x.ptr(6), x.ptr(7), x.nbytes(7))
ENTRY(recalibrate, 10, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), x.i32(4), x.i32(5), (float*)x.ptr(6),
      (float*)x.ptr(7), x.ptr(8), x.ptr(9), x.nbytes(9))
ENTRY(accumulated_scores, 5, x.params(0), x.ptr(1), x.ptr(2), (float*)x.ptr(3), x.ptr(4), x.nbytes(4))
ENTRY(select_from_scores, 5, x.params(0), (const float*)x.ptr(1), x.i32(2), (int32_t*)x.ptr(3), x.ptr(4), x.nbytes(4))
ENTRY(select_streaming, 3, x.params(0), x.i32(1), (int32_t*)x.ptr(2))
ENTRY(decode, 14, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), x.ptr(4), x.ptr(5), x.i32(6), (const float*)x.ptr(7),
      (const float*)x.ptr(8), x.ptr(9), x.ptr(10), (float*)x.ptr(11), (uint8_t*)x.ptr(12), x.ptr(13), x.nbytes(13))
ENTRY(decode_batched, 4, x.params(0), (int32_t)x.len(1), x.layers(1), x.i32(2), x.ptr(3),
      x.nbytes(3))
ENTRY(decode_static, 13, x.params(0), x.ptr(1), x.ptr(2), x.ptr(3), x.ptr(4), x.ptr(5), x.i32(6), (const float*)x.ptr(7),
      (const float*)x.ptr(8), x.ptr(9), x.ptr(10), (float*)x.ptr(11), (uint8_t*)x.ptr(12))

// open(path, Params, DecodeLayer): the shared library whose entry points the functions forward to, and the ctypes
// structures of its arguments
PyObject* py_open(PyObject*, PyObject* const* args, Py_ssize_t n) {
  if (n != 3 || !PyType_Check(args[1]) || !PyType_Check(args[2]))
    return PyErr_Format(PyExc_TypeError, "a path and two structure types expected");
  const char* s = PyUnicode_AsUTF8(args[0]);
  if (!s) return nullptr;
  for (int i = 1; i < 3; ++i) {
    PyObject* o = PyObject_CallNoArgs(args[i]);
    Py_buffer v;
    if (!o) return nullptr;
    const bool buffer = PyObject_GetBuffer(o, &v, PyBUF_SIMPLE) == 0;
    Py_DECREF(o);
    if (!buffer) return nullptr;
    const bool same = v.len == (Py_ssize_t)(i == 1 ? sizeof(calidrop_params) : sizeof(calidrop_decode_layer));
    PyBuffer_Release(&v);
    if (!same) return PyErr_Format(PyExc_TypeError, "the structure's size is not the library's");
  }
  void* h = dlopen(s, RTLD_NOW | RTLD_LOCAL);
  if (!h) return PyErr_Format(PyExc_ImportError, "%s", dlerror());
#define RESOLVE(name)                                                                               \
  f_##name = (decltype(f_##name))dlsym(h, "calidrop_" #name);                                        \
  if (!f_##name) return PyErr_Format(PyExc_ImportError, "%s does not export calidrop_" #name, s);
  CALIDROP_ENTRIES(RESOLVE)
#undef RESOLVE
  params_type = (PyTypeObject*)Py_NewRef(args[1]);
  layer_type = (PyTypeObject*)Py_NewRef(args[2]);
  Py_RETURN_NONE;
}

PyMethodDef methods[] = {
    {"open", (PyCFunction)(void (*)(void))py_open, METH_FASTCALL, nullptr},
#define METHOD(name) {#name, (PyCFunction)(void (*)(void))py_##name, METH_FASTCALL, nullptr},
    CALIDROP_ENTRIES(METHOD)
#undef METHOD
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal() { return PyModule_Create(&module); }
