// The calls of a decode step without ctypes: a Python extension that takes the arguments of the binding's methods
// (tensors, device addresses or None), makes the pointers of them and calls the C ABI with the interpreter lock released, as ctypes
// does.  An argument that it cannot convert is not judged here: the function returns NotImplemented and the binding goes through
// ctypes, which converts it or raises what it always raised.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/gkv.h"

namespace {

// the library's entry points, handed over by the binding, which has loaded it
decltype(&gkv_append_demote) f_append = nullptr;
decltype(&gkv_decode_attn) f_decode = nullptr;
decltype(&gkv_decode_attn_observe) f_observe = nullptr;
decltype(&gkv_quest_select) f_select = nullptr;
PyObject* s_data_ptr = nullptr;      // "data_ptr"
PyObject* s_value = nullptr;         // "value"
PyObject* void_p = nullptr;          // ctypes.c_void_p

// an int or None
bool as_plain(PyObject* o, void** out) {
  if (o != Py_None && !PyLong_Check(o)) return false;
  *out = o == Py_None ? nullptr : reinterpret_cast<void*>(static_cast<uintptr_t>(PyLong_AsUnsignedLongLongMask(o)));
  return !PyErr_Occurred();
}
// an int, None, or a tensor
bool as_address(PyObject* o, void** out) {
  if (o == Py_None || PyLong_Check(o)) return as_plain(o, out);
  PyObject* v = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!v) return false;
  const bool ok = as_plain(v, out);
  Py_DECREF(v);
  return ok;
}
// a ctypes.c_void_p, an int or None
bool as_handle(PyObject* o, gkv_cache** out) {
  void* p = nullptr;
  bool ok;
  if (reinterpret_cast<PyObject*>(Py_TYPE(o)) == void_p) {
    PyObject* v = PyObject_GetAttr(o, s_value);
    if (!v) return false;
    ok = as_plain(v, &p);
    Py_DECREF(v);
  } else {
    ok = as_plain(o, &p);
  }
  *out = static_cast<gkv_cache*>(p);
  return ok;
}
bool as_int(PyObject* o, int32_t* out) {
  if (!PyLong_Check(o)) return false;
  *out = static_cast<int32_t>(PyLong_AsUnsignedLongMask(o));
  return !PyErr_Occurred();
}
// An exception of the conversion is raised again, or not, by the binding's second attempt (an interrupt is not one).
PyObject* refuse() {
  if (PyErr_Occurred()) {
    if (!PyErr_ExceptionMatches(PyExc_Exception)) return nullptr;
    PyErr_Clear();
  }
  Py_RETURN_NOTIMPLEMENTED;
}
bool want(Py_ssize_t n, Py_ssize_t need) {
  if (n == need) return true;
  PyErr_Format(PyExc_TypeError, "%zd arguments are needed, not %zd", need, n);
  return false;
}

// bind(append, decode, observe, select, c_void_p): addresses, and ctypes' type of a handle
PyObject* py_bind(PyObject*, PyObject* const* a, Py_ssize_t n) {
  void* p[4];
  if (!want(n, 5)) return nullptr;
  for (int i = 0; i < 4; ++i)
    if (!as_plain(a[i], &p[i])) return PyErr_Occurred() ? nullptr : PyErr_Format(PyExc_TypeError, "an address is needed");
  Py_INCREF(a[4]);
  Py_XSETREF(void_p, a[4]);
  f_append = reinterpret_cast<decltype(f_append)>(p[0]);
  f_decode = reinterpret_cast<decltype(f_decode)>(p[1]);
  f_observe = reinterpret_cast<decltype(f_observe)>(p[2]);
  f_select = reinterpret_cast<decltype(f_select)>(p[3]);
  Py_RETURN_NONE;
}

// append(handle, layer, k, v, n_new, token_mass, level_plan, stream)
PyObject* py_append(PyObject*, PyObject* const* a, Py_ssize_t n) {
  gkv_cache* h;
  int32_t layer, n_new;
  void *k, *v, *mass, *plan, *st;
  if (!want(n, 8)) return nullptr;
  if (!as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_address(a[2], &k) || !as_address(a[3], &v) || !as_int(a[4], &n_new) ||
      !as_address(a[5], &mass) || !as_address(a[6], &plan) || !as_plain(a[7], &st))
    return refuse();
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_append(h, layer, k, v, n_new, static_cast<const float*>(mass), static_cast<const int8_t*>(plan), st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// decode(handle, layer, q, page_idx, n_sel, out, lse, stream)
PyObject* py_decode(PyObject*, PyObject* const* a, Py_ssize_t n) {
  gkv_cache* h;
  int32_t layer, n_sel;
  void *q, *pages, *out, *lse, *st;
  if (!want(n, 8)) return nullptr;
  if (!as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_address(a[2], &q) || !as_address(a[3], &pages) || !as_int(a[4], &n_sel) ||
      !as_address(a[5], &out) || !as_address(a[6], &lse) || !as_plain(a[7], &st))
    return refuse();
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_decode(h, layer, q, static_cast<const int32_t*>(pages), n_sel, static_cast<float*>(out), static_cast<float*>(lse), st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// observe(handle, layer, q, out, lse, block_mass, certificate, stream)
PyObject* py_observe(PyObject*, PyObject* const* a, Py_ssize_t n) {
  gkv_cache* h;
  int32_t layer;
  void *q, *out, *lse, *mass, *cert, *st;
  if (!want(n, 8)) return nullptr;
  if (!as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_address(a[2], &q) || !as_address(a[3], &out) || !as_address(a[4], &lse) ||
      !as_address(a[5], &mass) || !as_address(a[6], &cert) || !as_plain(a[7], &st))
    return refuse();
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_observe(h, layer, q, static_cast<float*>(out), static_cast<float*>(lse), static_cast<float*>(mass), static_cast<float*>(cert), st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// select(handle, layer, q, budget_tokens, page_idx_out, stream) -> (status, pages selected)
PyObject* py_select(PyObject*, PyObject* const* a, Py_ssize_t n) {
  gkv_cache* h;
  int32_t layer, budget, n_sel = 0;
  void *q, *pages, *st;
  if (!want(n, 6)) return nullptr;
  if (!as_handle(a[0], &h) || !as_int(a[1], &layer) || !as_address(a[2], &q) || !as_int(a[3], &budget) || !as_address(a[4], &pages) ||
      !as_plain(a[5], &st))
    return refuse();
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_select(h, layer, q, budget, static_cast<int32_t*>(pages), &n_sel, st);
  Py_END_ALLOW_THREADS
  return Py_BuildValue("(ii)", rc, static_cast<int>(n_sel));
}

#define GKV_FAST(name, f) {name, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {GKV_FAST("bind", py_bind),       GKV_FAST("append", py_append), GKV_FAST("decode", py_decode),
                         GKV_FAST("observe", py_observe), GKV_FAST("select", py_select), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_gkv_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__gkv_call() {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_value = PyUnicode_InternFromString("value");
  return s_data_ptr && s_value ? PyModule_Create(&module) : nullptr;
}
