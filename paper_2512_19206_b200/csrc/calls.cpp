// The calls of a decode step without ctypes: argument marshalling for CPython, nothing else.
//
// A call on a small cache is bound by the host: its kernels take 3 to 4 us and the launch about 2.  ctypes converts ten
// arguments in 2.6 us (measured on a null handle) and the address of a tensor costs 0.4 us of Python; here both
// are a few attribute lookups in C (0.15 us on the null handle).  decode_attention on one sequence of 1024 tokens, calls
// one after the other: 6.30 -> 5.26 us; calls whose GPU work is longer than the host's are unchanged.  Only the calls that a generation loop makes per layer and token are here; the
// others move enough data for ctypes not to matter.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/mixkvq.h"

namespace {

PyObject *s_is_cuda, *s_is_contiguous, *s_data_ptr;

// Handle and stream: an int, or None for a null pointer.
bool raw(PyObject* o, void** p) {
  *p = o == Py_None ? nullptr : PyLong_AsVoidPtr(o);
  return *p || !PyErr_Occurred();
}

// The address of a contiguous CUDA tensor (None: a null pointer, which the library refuses).
bool address(PyObject* o, void** p) {
  if (o == Py_None) {
    *p = nullptr;
    return true;
  }
  PyObject* x = PyObject_GetAttr(o, s_is_cuda);
  if (!x) return false;
  int yes = PyObject_IsTrue(x);
  Py_DECREF(x);
  if (yes > 0) {
    x = PyObject_CallMethodNoArgs(o, s_is_contiguous);
    if (!x) return false;
    yes = PyObject_IsTrue(x);
    Py_DECREF(x);
  }
  if (yes < 0) return false;
  if (!yes) {
    PyErr_SetString(PyExc_AssertionError, "a contiguous CUDA tensor is needed");
    return false;
  }
  x = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!x) return false;
  *p = PyLong_AsVoidPtr(x);
  Py_DECREF(x);
  return *p || !PyErr_Occurred();
}

bool integer(PyObject* o, int* i) {
  *i = static_cast<int>(PyLong_AsUnsignedLongMask(o));
  return !PyErr_Occurred();
}

bool size(PyObject* o, size_t* n) {
  *n = PyLong_AsSize_t(o);
  return !PyErr_Occurred();
}

bool real(PyObject* o, float* f) {
  if (PyFloat_CheckExact(o)) {
    *f = static_cast<float>(PyFloat_AS_DOUBLE(o));
    return true;
  }
  PyObject* x = PyNumber_Float(o);
  if (!x) return false;
  *f = static_cast<float>(PyFloat_AS_DOUBLE(x));
  Py_DECREF(x);
  return true;
}

bool count_is(Py_ssize_t n, Py_ssize_t want) {
  if (n != want) PyErr_Format(PyExc_TypeError, "%zd arguments are needed, %zd were given", want, n);
  return n == want;
}

mixkvq_cache* cache_of(void* p) { return static_cast<mixkvq_cache*>(p); }

// (handle, layer, q, out, scale, workspace, workspace bytes, stream)
PyObject* decode_attention(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *h, *q, *out, *ws, *st;
  int layer, rc;
  float scale;
  size_t bytes;
  if (!count_is(n, 8) || !raw(a[0], &h) || !integer(a[1], &layer) || !address(a[2], &q) || !address(a[3], &out) ||
      !real(a[4], &scale) || !address(a[5], &ws) || !size(a[6], &bytes) || !raw(a[7], &st))
    return nullptr;
  Py_BEGIN_ALLOW_THREADS
  rc = mixkvq_decode_attention(cache_of(h), layer, q, static_cast<float*>(out), scale, ws, bytes, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (handle, layer, k, v, q, out, scale, workspace, workspace bytes, stream)
PyObject* decode_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *h, *k, *v, *q, *out, *ws, *st;
  int layer, rc;
  float scale;
  size_t bytes;
  if (!count_is(n, 10) || !raw(a[0], &h) || !integer(a[1], &layer) || !address(a[2], &k) || !address(a[3], &v) ||
      !address(a[4], &q) || !address(a[5], &out) || !real(a[6], &scale) || !address(a[7], &ws) || !size(a[8], &bytes) ||
      !raw(a[9], &st))
    return nullptr;
  Py_BEGIN_ALLOW_THREADS
  rc = mixkvq_decode_step(cache_of(h), layer, k, v, q, static_cast<float*>(out), scale, ws, bytes, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (handle, layer, k, v, q, cos, sin, position, out, scale, workspace, workspace bytes, stream)
PyObject* rope_decode_step(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *h, *k, *v, *q, *cos, *sin, *out, *ws, *st;
  int layer, pos, rc;
  float scale;
  size_t bytes;
  if (!count_is(n, 13) || !raw(a[0], &h) || !integer(a[1], &layer) || !address(a[2], &k) || !address(a[3], &v) ||
      !address(a[4], &q) || !address(a[5], &cos) || !address(a[6], &sin) || !integer(a[7], &pos) ||
      !address(a[8], &out) || !real(a[9], &scale) || !address(a[10], &ws) || !size(a[11], &bytes) ||
      !raw(a[12], &st))
    return nullptr;
  Py_BEGIN_ALLOW_THREADS
  rc = mixkvq_rope_decode_step(cache_of(h), layer, k, v, q, static_cast<const float*>(cos), static_cast<const float*>(sin),
                               pos, static_cast<float*>(out), scale, ws, bytes, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (handle, layer, k, v, q, tokens, stream)
PyObject* quantize_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void *h, *k, *v, *q, *st;
  int layer, tokens, rc;
  if (!count_is(n, 7) || !raw(a[0], &h) || !integer(a[1], &layer) || !address(a[2], &k) || !address(a[3], &v) ||
      !address(a[4], &q) || !integer(a[5], &tokens) || !raw(a[6], &st))
    return nullptr;
  Py_BEGIN_ALLOW_THREADS
  rc = mixkvq_quantize_append(cache_of(h), layer, k, v, q, tokens, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

template <typename F>
PyCFunction fast(F f) {
  return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f));
}

PyMethodDef methods[] = {{"decode_attention", fast(decode_attention), METH_FASTCALL, nullptr},
                         {"decode_step", fast(decode_step), METH_FASTCALL, nullptr},
                         {"rope_decode_step", fast(rope_decode_step), METH_FASTCALL, nullptr},
                         {"quantize_append", fast(quantize_append), METH_FASTCALL, nullptr},
                         {nullptr, nullptr, 0, nullptr}};

PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__calls() {
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  if (!s_is_cuda || !s_is_contiguous || !s_data_ptr) return nullptr;
  return PyModule_Create(&module);
}
