/* The two calls of a generated token (lrsa_cache_append, lrsa_attn_decode) as a Python module over plain integers: both are
 * host-bound for one sequence, and a foreign-function call with ten arguments takes 1.1 us where this takes 0.2.  Every
 * other entry point goes through ctypes. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "../../include/lrsa.h"

/* args[i] as an address, a size or a count; None is a null pointer */
static unsigned long long arg(PyObject* const* args, int i) {
  return args[i] == Py_None ? 0ull : PyLong_AsUnsignedLongLong(args[i]);
}
#define PTR(i) ((void*)(uintptr_t)arg(args, i))

/* (params, cache, cache_bytes, k_new, v_new, n_prev, n_new, workspace, workspace_bytes, stream) -> status */
static PyObject* cache_append(PyObject* self, PyObject* const* args, Py_ssize_t n) {
  (void)self;
  if (n != 10) return PyErr_Format(PyExc_TypeError, "cache_append takes 10 arguments");
  const lrsa_params_t* p = (const lrsa_params_t*)PTR(0);
  void *cache = PTR(1), *k = PTR(3), *v = PTR(4), *ws = PTR(7), *st = PTR(9);
  const size_t bytes = (size_t)arg(args, 2), ws_bytes = (size_t)arg(args, 8);
  const int32_t n_prev = (int32_t)PyLong_AsLong(args[5]), n_new = (int32_t)PyLong_AsLong(args[6]);
  if (PyErr_Occurred()) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = lrsa_cache_append(p, cache, bytes, k, v, n_prev, n_new, ws, ws_bytes, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* (params, cache, cache_bytes, q, n_tokens, o, lse, workspace, workspace_bytes, stream) -> status */
static PyObject* attn_decode(PyObject* self, PyObject* const* args, Py_ssize_t n) {
  (void)self;
  if (n != 10) return PyErr_Format(PyExc_TypeError, "attn_decode takes 10 arguments");
  const lrsa_params_t* p = (const lrsa_params_t*)PTR(0);
  void *cache = PTR(1), *q = PTR(3), *o = PTR(5), *lse = PTR(6), *ws = PTR(7), *st = PTR(9);
  const size_t bytes = (size_t)arg(args, 2), ws_bytes = (size_t)arg(args, 8);
  const int32_t n_tokens = (int32_t)PyLong_AsLong(args[4]);
  if (PyErr_Occurred()) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = lrsa_attn_decode(p, cache, bytes, q, n_tokens, o, (float*)lse, ws, ws_bytes, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"cache_append", (PyCFunction)(void (*)(void))cache_append, METH_FASTCALL, NULL},
    {"attn_decode", (PyCFunction)(void (*)(void))attn_decode, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_lrsa_call", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__lrsa_call(void) { return PyModule_Create(&module); }
