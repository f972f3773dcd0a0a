// CPython face of the four codec calls of include/tahq.h.  A call through ctypes spends two to three microseconds on
// building the parameter structure and converting arguments, as long as the launch itself; here the structure comes
// as the bytes that the caller keeps, and the arguments are integers taken one by one.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <string.h>

#include <initializer_list>

#include "../../include/tahq.h"

namespace {

// An address or a size: a Python integer (taken modulo 2^64), or None for a null pointer; else what ctypes would take, a
// c_void_p or c_size_t by its value, and an object with an `_as_parameter_` (a torch stream has one).
bool to_word(PyObject *o, unsigned long long *v) {
  if (o == Py_None) { *v = 0; return true; }
  if (PyLong_Check(o)) {
    *v = PyLong_AsUnsignedLongLongMask(o);
    return !(*v == (unsigned long long)-1 && PyErr_Occurred());
  }
  for (const char *name : {"_as_parameter_", "value"}) {
    PyObject *w = PyObject_GetAttrString(o, name);
    if (!w) {
      if (!PyErr_ExceptionMatches(PyExc_AttributeError)) return false;
      PyErr_Clear();
      continue;
    }
    bool ok = false;
    if (w == Py_None || PyLong_Check(w)) {
      ok = to_word(w, v);
    } else {   // (a stream's parameter is a c_void_p)
      PyObject *x = PyObject_GetAttrString(w, "value");
      if (x && (x == Py_None || PyLong_Check(x))) ok = to_word(x, v);
      else PyErr_Format(PyExc_TypeError, "expected an integer or None, got %.100s", Py_TYPE(w)->tp_name);
      Py_XDECREF(x);
    }
    Py_DECREF(w);
    return ok;
  }
  PyErr_Format(PyExc_TypeError, "expected an integer or None, got %.100s", Py_TYPE(o)->tp_name);
  return false;
}

// (params: bytes, six words): pointer, pointer or size ... in the order of the C function
template <class P, class F>
PyObject *call(PyObject *const *args, Py_ssize_t n, F &&f) {
  if (n != 7) { PyErr_SetString(PyExc_TypeError, "expected the parameters and six integers"); return nullptr; }
  if (!PyBytes_Check(args[0]) || PyBytes_GET_SIZE(args[0]) != (Py_ssize_t)sizeof(P)) {
    PyErr_SetString(PyExc_TypeError, "expected the bytes of the parameter structure");
    return nullptr;
  }
  P p;
  memcpy(&p, PyBytes_AS_STRING(args[0]), sizeof(p));
  unsigned long long w[6];
  for (int i = 0; i < 6; ++i)
    if (!to_word(args[i + 1], &w[i])) return nullptr;
  tahq_status s;
  Py_BEGIN_ALLOW_THREADS   // a launch may wait for room in the stream's queue
  s = f(p, w);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)s);
}
void *ptr(unsigned long long v) { return reinterpret_cast<void *>(static_cast<uintptr_t>(v)); }
tahq_stream stream(unsigned long long v) { return static_cast<tahq_stream>(ptr(v)); }

PyObject *encode(PyObject *, PyObject *const *args, Py_ssize_t n) {
  return call<tahq_params>(args, n, [](const tahq_params &p, const unsigned long long *w) {
    return tahq_encode(&p, ptr(w[0]), ptr(w[1]), w[2], ptr(w[3]), w[4], stream(w[5]));
  });
}
PyObject *decode(PyObject *, PyObject *const *args, Py_ssize_t n) {
  return call<tahq_params>(args, n, [](const tahq_params &p, const unsigned long long *w) {
    return tahq_decode(&p, ptr(w[0]), w[1], ptr(w[2]), ptr(w[3]), w[4], stream(w[5]));
  });
}
PyObject *qnaive_encode(PyObject *, PyObject *const *args, Py_ssize_t n) {
  return call<tahq_qnaive_params>(args, n, [](const tahq_qnaive_params &p, const unsigned long long *w) {
    return tahq_qnaive_encode(&p, ptr(w[0]), ptr(w[1]), w[2], ptr(w[3]), w[4], stream(w[5]));
  });
}
PyObject *qnaive_decode(PyObject *, PyObject *const *args, Py_ssize_t n) {
  return call<tahq_qnaive_params>(args, n, [](const tahq_qnaive_params &p, const unsigned long long *w) {
    return tahq_qnaive_decode(&p, ptr(w[0]), w[1], ptr(w[2]), ptr(w[3]), w[4], stream(w[5]));
  });
}

PyCFunction method(PyObject *(*f)(PyObject *, PyObject *const *, Py_ssize_t)) {
  return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f));
}
PyMethodDef methods[] = {
    {"encode", method(encode), METH_FASTCALL,
     "encode(params, d_in, d_packed, packed_cap, d_ws, ws_cap, stream) -> tahq_status"},
    {"decode", method(decode), METH_FASTCALL,
     "decode(params, d_packed, packed_bytes, d_out, d_ws, ws_cap, stream) -> tahq_status"},
    {"qnaive_encode", method(qnaive_encode), METH_FASTCALL,
     "qnaive_encode(params, d_in, d_packed, packed_cap, d_ws, ws_cap, stream) -> tahq_status"},
    {"qnaive_decode", method(qnaive_decode), METH_FASTCALL,
     "qnaive_decode(params, d_packed, packed_bytes, d_out, d_ws, ws_cap, stream) -> tahq_status"},
    {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__call(void) { return PyModule_Create(&module); }
