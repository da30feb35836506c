/* Argument marshalling of the per-step calls for the Python binding.
 *
 * Through ctypes a call spends most of its host time converting arguments and
 * reading array addresses: more than the GPU takes for a short step or for one
 * layer of a small batch.  Here a call converts its arguments with the C API
 * and calls the library directly.  On a Grace core, a decode step and its
 * observation: 448 tokens 26.0 -> 15.8 us, 1,700 tokens 32.9 -> 18.8 us; 28
 * layer calls 176 -> 143 us.
 *
 * Device buffers are None, an address, or an object with data_ptr() (a torch
 * tensor).  Host arrays are taken in place when they are C-contiguous of the
 * exact type; for anything else a call returns None and the caller converts
 * the array first.  The GIL is released around the library's calls, as ctypes
 * does. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <dlfcn.h>

#include "../../include/memdecay.h"

static PyObject *s_data_ptr, *s_is_cuda, *s_is_contiguous;
static md_status (*f_decode_step)(md_ctx *, int, const void *, const void *, const void *, const uint8_t *, void *);
static md_status (*f_decode_step_host)(md_ctx *, int, const void *, const void *, const void *, const uint8_t *,
                                       void *);
static md_status (*f_decode_layer)(md_ctx *, int, int, const void *, const void *, const void *, const uint8_t *,
                                   void *);
static md_status (*f_evict)(md_ctx *, int, const int32_t *, int32_t *, int32_t *);
static md_status (*f_get_state)(md_ctx *, int, void *, size_t);

static PyObject *load(PyObject *self, PyObject *path) {
  const char *s = PyUnicode_AsUTF8(path);
  if (!s) return NULL;
  void *h = dlopen(s, RTLD_NOW | RTLD_LOCAL);
  if (!h) {
    PyErr_SetString(PyExc_OSError, dlerror());
    return NULL;
  }
  *(void **)&f_decode_step = dlsym(h, "md_decode_step");
  *(void **)&f_decode_step_host = dlsym(h, "md_decode_step_host");
  *(void **)&f_decode_layer = dlsym(h, "md_decode_layer");
  *(void **)&f_evict = dlsym(h, "md_evict");
  *(void **)&f_get_state = dlsym(h, "md_get_state");
  if (!f_decode_step || !f_decode_step_host || !f_decode_layer || !f_evict || !f_get_state) {
    PyErr_SetString(PyExc_OSError, "libmemdecay.so lacks an entry point");
    return NULL;
  }
  Py_RETURN_NONE;
}

/* Device address of a buffer argument; -1 with an exception set on failure. */
static int dev_ptr(PyObject *o, void **out) {
  if (o == Py_None) {
    *out = NULL;
    return 0;
  }
  if (PyLong_Check(o)) {
    *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(o);
    return PyErr_Occurred() ? -1 : 0;
  }
  PyObject *v = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (!v) return -1;
  *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

/* Address of a contiguous CPU tensor: 1, 0 if it is something else or not
 * contiguous (no exception: the caller reports it), -1 with an exception. */
static int host_ptr(PyObject *o, void **out) {
  PyObject *v = PyObject_GetAttr(o, s_is_cuda);
  if (!v) {
    PyErr_Clear();
    return 0;
  }
  const int cuda = v != Py_False;
  Py_DECREF(v);
  if (cuda) return 0;
  v = PyObject_CallMethodNoArgs(o, s_is_contiguous);
  if (!v) return -1;
  const int dense = v == Py_True;
  Py_DECREF(v);
  if (!dense) return 0;
  return dev_ptr(o, out) ? -1 : 1;
}

/* A one-dimensional C-contiguous buffer of items with this format: 1 and the
 * view (to be released), 0 if it is something else, never an exception.  Not a
 * byte string: the caller's conversion reads its bytes as text. */
static int host_view(PyObject *o, char format, Py_ssize_t item, int writable, Py_buffer *view) {
  if (PyBytes_Check(o)) return 0;
  if (PyObject_GetBuffer(o, view, PyBUF_C_CONTIGUOUS | PyBUF_FORMAT | (writable ? PyBUF_WRITABLE : 0)) != 0) {
    PyErr_Clear();
    return 0;
  }
  const char *f = view->format ? view->format : "B";
  if (view->ndim == 1 && view->itemsize == item && f[0] == format && f[1] == 0) return 1;
  PyBuffer_Release(view);
  return 0;
}

/* The labels of a step: one per sequence of the batch at least. */
static int label_view(PyObject *o, int batch, Py_buffer *view) {
  if (!host_view(o, 'B', 1, 0, view)) return 0;
  if (view->shape[0] >= batch) return 1;
  PyBuffer_Release(view);
  return 0;
}

static int as_int(PyObject *o, int *out) {
  const long long v = PyLong_AsLongLong(o);
  if (v == -1 && PyErr_Occurred()) return -1;
  *out = (int)v;
  return 0;
}

static int arity(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return 0;
  PyErr_SetString(PyExc_TypeError, "wrong number of arguments");
  return -1;
}

/* decode_step(handle, batch, q, k_new, v_new, new_regions, out) -> status, or
 * None when new_regions must be converted */
static PyObject *decode_step(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *q, *k, *v, *out;
  int batch, st;
  Py_buffer regs;
  if (arity(n, 7) || dev_ptr(a[0], &h) || as_int(a[1], &batch) || dev_ptr(a[2], &q) || dev_ptr(a[3], &k) ||
      dev_ptr(a[4], &v) || dev_ptr(a[6], &out))
    return NULL;
  if (!label_view(a[5], batch, &regs)) Py_RETURN_NONE;
  Py_BEGIN_ALLOW_THREADS
  st = f_decode_step((md_ctx *)h, batch, q, k, v, (const uint8_t *)regs.buf, out);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&regs);
  return PyLong_FromLong(st);
}

/* decode_step_host(handle, batch, q, k_new, v_new, new_regions, out): host
 * buffers are contiguous CPU tensors */
static PyObject *decode_step_host(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *x[4];
  int batch, st;
  Py_buffer regs;
  if (arity(n, 7) || dev_ptr(a[0], &h) || as_int(a[1], &batch)) return NULL;
  for (int i = 0; i < 4; ++i) {
    const int ok = host_ptr(a[i < 3 ? 2 + i : 6], &x[i]);
    if (ok < 0) return NULL;
    if (ok == 0) Py_RETURN_NONE;
  }
  if (!label_view(a[5], batch, &regs)) Py_RETURN_NONE;
  Py_BEGIN_ALLOW_THREADS
  st = f_decode_step_host((md_ctx *)h, batch, x[0], x[1], x[2], (const uint8_t *)regs.buf, x[3]);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&regs);
  return PyLong_FromLong(st);
}

/* decode_layer(handle, layer, batch, q, k_new, v_new, new_regions, out) */
static PyObject *decode_layer(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *q, *k, *v, *out;
  int layer, batch, st;
  Py_buffer regs;
  if (arity(n, 8) || dev_ptr(a[0], &h) || as_int(a[1], &layer) || as_int(a[2], &batch) || dev_ptr(a[3], &q) ||
      dev_ptr(a[4], &k) || dev_ptr(a[5], &v) || dev_ptr(a[7], &out))
    return NULL;
  if (!label_view(a[6], layer == 0 ? batch : 0, &regs)) Py_RETURN_NONE;   // later layers read none
  Py_BEGIN_ALLOW_THREADS
  st = f_decode_layer((md_ctx *)h, layer, batch, q, k, v, (const uint8_t *)regs.buf, out);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&regs);
  return PyLong_FromLong(st);
}

/* evict(handle, budgets, n_evicted, evicted_ids) -> status; budgets and
 * n_evicted are int32 arrays of one length, or None is returned */
static PyObject *evict(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *ids;
  int st;
  Py_buffer bud, ev;
  if (arity(n, 4) || dev_ptr(a[0], &h) || dev_ptr(a[3], &ids)) return NULL;
  if (!host_view(a[1], 'i', 4, 0, &bud)) Py_RETURN_NONE;
  if (!host_view(a[2], 'i', 4, 1, &ev)) {
    PyBuffer_Release(&bud);
    Py_RETURN_NONE;
  }
  if (bud.shape[0] != ev.shape[0]) {
    PyBuffer_Release(&bud);
    PyBuffer_Release(&ev);
    Py_RETURN_NONE;
  }
  Py_BEGIN_ALLOW_THREADS
  st = f_evict((md_ctx *)h, (int)bud.shape[0], (const int32_t *)bud.buf, (int32_t *)ev.buf, (int32_t *)ids);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&bud);
  PyBuffer_Release(&ev);
  return PyLong_FromLong(st);
}

/* get_state(handle, what, dst, bytes) -> status */
static PyObject *get_state(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  void *h, *dst;
  int what, st;
  if (arity(n, 4) || dev_ptr(a[0], &h) || as_int(a[1], &what) || dev_ptr(a[2], &dst)) return NULL;
  const long long bytes = PyLong_AsLongLong(a[3]);
  if (bytes == -1 && PyErr_Occurred()) return NULL;
  Py_BEGIN_ALLOW_THREADS
  st = f_get_state((md_ctx *)h, what, dst, (size_t)bytes);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

static PyMethodDef methods[] = {
    {"load", load, METH_O, "load(path): binds the calls to libmemdecay.so"},
    {"decode_step", (PyCFunction)(void (*)(void))decode_step, METH_FASTCALL, "md_decode_step"},
    {"decode_step_host", (PyCFunction)(void (*)(void))decode_step_host, METH_FASTCALL, "md_decode_step_host"},
    {"decode_layer", (PyCFunction)(void (*)(void))decode_layer, METH_FASTCALL, "md_decode_layer"},
    {"evict", (PyCFunction)(void (*)(void))evict, METH_FASTCALL, "md_evict"},
    {"get_state", (PyCFunction)(void (*)(void))get_state, METH_FASTCALL, "md_get_state"},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  return s_data_ptr && s_is_cuda && s_is_contiguous ? PyModule_Create(&module) : NULL;
}
