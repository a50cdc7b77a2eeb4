/* CPython entry to the calls a program makes per step.
 *
 * Through ctypes a call of seven arguments costs about two microseconds of argument conversion and list building, as much as a
 * kernel launch; a chain that is one small copy spends more time there than on the device.  These functions take the same
 * arguments, convert them directly and call the library through the addresses `bind` was given.  The GIL is released around
 * the call, as ctypes does.  They take the plain forms only -- a parameter block of the type `bind` was given, addresses as int or
 * None, lists or tuples of them -- and return None, nothing called, for everything else: the caller then goes through ctypes, which
 * accepts or refuses it. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*swin_fn)(const void*, const void*, void*, void*, size_t, int32_t, void*);
typedef int (*attn_fn)(const void*, const void*, void*, void*, size_t, int32_t, void*);
typedef int (*decode_fn)(const void*, int32_t, const void*, void*, void*, void*, void*, size_t, int32_t, void*);
typedef int (*chain_fn)(const void*, const void* const*, void* const*, void*, size_t, void*);
static swin_fn g_swin;
static attn_fn g_attn;
static decode_fn g_decode;
static chain_fn g_chain;
static PyTypeObject *g_swin_type, *g_attn_type;     /* the parameter blocks: ctypes structures */

#define MAX_PTRS 16

/* an address: an int or None (null) */
static int as_ptr(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = NULL;
    return 1;
  }
  *out = PyLong_AsVoidPtr(o);
  return !(*out == NULL && PyErr_Occurred());
}
static int as_size(PyObject* o, size_t* out) {
  *out = PyLong_AsSize_t(o);
  return !(*out == (size_t)-1 && PyErr_Occurred());
}
static int as_int(PyObject* o, int32_t* out) {
  const long v = PyLong_AsLong(o);
  if (v == -1 && PyErr_Occurred()) return 0;
  *out = (int32_t)v;
  return 1;
}
static PyObject* not_plain(void) {
  PyErr_Clear();
  Py_RETURN_NONE;
}
/* the bytes of a parameter block of that type */
static int as_block(PyObject* o, PyTypeObject* type, Py_buffer* p) { return PyObject_TypeCheck(o, type) && !PyObject_GetBuffer(o, p, PyBUF_SIMPLE); }

/* (addresses of the four calls, types of the two parameter blocks) */
static PyObject* bind(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *s, *l, *d, *c;
  if (n != 6 || !PyType_Check(a[4]) || !PyType_Check(a[5])) {
    PyErr_SetString(PyExc_TypeError, "four addresses and two types are expected");
    return NULL;
  }
  if (!as_ptr(a[0], &s) || !as_ptr(a[1], &l) || !as_ptr(a[2], &d) || !as_ptr(a[3], &c)) return NULL;
  Py_INCREF(a[4]);
  Py_INCREF(a[5]);
  Py_XDECREF(g_swin_type);
  Py_XDECREF(g_attn_type);
  g_swin_type = (PyTypeObject*)a[4];
  g_attn_type = (PyTypeObject*)a[5];
  g_swin = (swin_fn)s;
  g_attn = (attn_fn)l;
  g_decode = (decode_fn)d;
  g_chain = (chain_fn)c;
  Py_RETURN_NONE;
}

/* (params, x, y, workspace, workspace_bytes, mode, stream) */
static PyObject* layer_call(swin_fn fn, PyTypeObject* type, PyObject* const* a, Py_ssize_t n) {
  void *x, *y, *ws, *st;
  size_t bytes;
  int32_t mode, rc;
  Py_buffer p;
  if (n != 7 || !type || !as_ptr(a[1], &x) || !as_ptr(a[2], &y) || !as_ptr(a[3], &ws) || !as_size(a[4], &bytes) || !as_int(a[5], &mode) ||
      !as_ptr(a[6], &st) || !as_block(a[0], type, &p))
    return not_plain();
  Py_BEGIN_ALLOW_THREADS
  rc = fn(p.buf, x, y, ws, bytes, mode, st);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&p);
  return PyLong_FromLong(rc);
}
static PyObject* swin_block(PyObject* self, PyObject* const* a, Py_ssize_t n) { return layer_call(g_swin, g_swin_type, a, n); }
static PyObject* attn_layer(PyObject* self, PyObject* const* a, Py_ssize_t n) { return layer_call(g_attn, g_attn_type, a, n); }

/* (params, pos, x, k_cache, v_cache, y, workspace, workspace_bytes, mode, stream) */
static PyObject* attn_decode(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *x, *k, *v, *y, *ws, *st;
  size_t bytes;
  int32_t pos, mode, rc;
  Py_buffer p;
  if (n != 10 || !g_attn_type || !as_int(a[1], &pos) || !as_ptr(a[2], &x) || !as_ptr(a[3], &k) || !as_ptr(a[4], &v) || !as_ptr(a[5], &y) ||
      !as_ptr(a[6], &ws) || !as_size(a[7], &bytes) || !as_int(a[8], &mode) || !as_ptr(a[9], &st) ||
      !as_block(a[0], g_attn_type, &p))
    return not_plain();
  Py_BEGIN_ALLOW_THREADS
  rc = g_decode(p.buf, pos, x, k, v, y, ws, bytes, mode, st);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&p);
  return PyLong_FromLong(rc);
}

/* the addresses of a list, in `small` or (long lists) in memory the caller frees when it differs from `small` */
static void** as_ptrs(PyObject* o, void** small) {
  if (!PyList_Check(o) && !PyTuple_Check(o)) return NULL;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(o);
  void** p = n <= MAX_PTRS ? small : PyMem_Malloc((size_t)n * sizeof(void*));
  if (!p) PyErr_NoMemory();
  for (Py_ssize_t i = 0; p && i < n; ++i)
    if (!as_ptr(PySequence_Fast_GET_ITEM(o, i), &p[i])) {
      if (p != small) PyMem_Free(p);
      p = NULL;
    }
  return p;
}

/* (plan, inputs, outputs, workspace, workspace_bytes, stream) */
static PyObject* run_chain(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *plan, *ws, *st, *in_s[MAX_PTRS] = {NULL}, *out_s[MAX_PTRS] = {NULL}, **in = in_s, **out = out_s;
  size_t bytes;
  int32_t rc = 0;
  int ok = n == 6 && g_chain && as_ptr(a[0], &plan) && (in = as_ptrs(a[1], in_s)) && (out = as_ptrs(a[2], out_s)) && as_ptr(a[3], &ws) &&
           as_size(a[4], &bytes) && as_ptr(a[5], &st);
  if (ok) {
    Py_BEGIN_ALLOW_THREADS
    rc = g_chain(plan, (const void* const*)in, out, ws, bytes, st);
    Py_END_ALLOW_THREADS
  }
  if (in && in != in_s) PyMem_Free(in);
  if (out && out != out_s) PyMem_Free(out);
  return ok ? PyLong_FromLong(rc) : not_plain();
}

static PyMethodDef methods[] = {{"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, NULL},
                                {"swin_block", (PyCFunction)(void (*)(void))swin_block, METH_FASTCALL, NULL},
                                {"attn_layer", (PyCFunction)(void (*)(void))attn_layer, METH_FASTCALL, NULL},
                                {"attn_decode", (PyCFunction)(void (*)(void))attn_decode, METH_FASTCALL, NULL},
                                {"run_chain", (PyCFunction)(void (*)(void))run_chain, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};
PyMODINIT_FUNC PyInit__fastcall(void) { return PyModule_Create(&module); }
