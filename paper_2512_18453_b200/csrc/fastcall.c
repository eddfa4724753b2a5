/* The binding's hot calls as a CPython extension: tensor checks, pointers, sizes and the current stream are
 * collected here instead of attribute by attribute in Python and through ctypes.  A three-kernel layer call spends
 * 7 us in its launches; the Python and ctypes work around it took 3.1 us, this takes 0.9 (a 16 x 16 layer in one
 * kernel: 5.9 -> 3.9 us per call).  The library's functions arrive as addresses, so that there is one copy of libnova. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "nova.h"

static struct {
  __typeof__(&nova_conv2d_fwd) conv2d;
  __typeof__(&nova_filter_transform) filter;
  __typeof__(&nova_conv2d_fwd_int8) int8;
} fn;
static PyObject *get_device, *get_stream;                 /* torch's accessors of the current device and stream */
static PyObject *s_is_cuda, *s_is_contiguous, *s_dtype, *s_shape, *s_data_ptr, *s_numel;

/* 1 if `t` is a contiguous CUDA tensor of `dtype`; 0 with AssertionError set, or -1 with another error */
static int check(PyObject* t, PyObject* dtype) {
  PyObject* v = PyObject_GetAttr(t, s_is_cuda);
  if (!v) return -1;
  int ok = v == Py_True;
  Py_DECREF(v);
  if (ok) {
    if (!(v = PyObject_CallMethodNoArgs(t, s_is_contiguous))) return -1;
    ok = v == Py_True;
    Py_DECREF(v);
  }
  if (ok) {
    if (!(v = PyObject_GetAttr(t, s_dtype))) return -1;
    ok = v == dtype;
    Py_DECREF(v);
  }
  if (!ok) PyErr_SetString(PyExc_AssertionError, "a contiguous CUDA tensor of the plan's storage type is needed");
  return ok;
}
/* the first `count` sizes of a tensor; `exact`: it has no more dimensions */
static int shape(PyObject* t, long long* out, Py_ssize_t count, int exact) {
  PyObject* s = PyObject_GetAttr(t, s_shape);
  if (!s) return 0;
  int ok = PyTuple_Check(s) && (exact ? PyTuple_GET_SIZE(s) == count : PyTuple_GET_SIZE(s) >= count);
  for (Py_ssize_t i = 0; ok && i < count; ++i) {
    out[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(s, i));
    if (out[i] < 0 || out[i] > INT32_MAX) ok = 0;
  }
  Py_DECREF(s);
  if (!ok && !PyErr_Occurred()) PyErr_Format(PyExc_ValueError, "a tensor of %zd dimensions is needed", count);
  return ok;
}
static int integer(PyObject* t, PyObject* method, unsigned long long* out) {
  PyObject* v = PyObject_CallMethodNoArgs(t, method);
  if (!v) return 0;
  *out = PyLong_AsUnsignedLongLong(v);
  Py_DECREF(v);
  return !PyErr_Occurred();
}
static int pointer(PyObject* t, void** out) {
  unsigned long long v;
  if (!integer(t, s_data_ptr, &v)) return 0;
  *out = (void*)(uintptr_t)v;
  return 1;
}
static int stream(nova_stream* out) {
  PyObject* dev = PyObject_CallNoArgs(get_device);
  if (!dev) return 0;
  PyObject* s = PyObject_CallOneArg(get_stream, dev);
  Py_DECREF(dev);
  if (!s) return 0;
  *out = (nova_stream)(uintptr_t)PyLong_AsUnsignedLongLong(s);
  Py_DECREF(s);
  return !PyErr_Occurred();
}

/* conv2d(plan, dtype, x, U, y, workspace, flags) -> status */
static PyObject* conv2d(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  long long d[4], u[2];
  void *x, *U, *y, *ws;
  unsigned long long bytes;
  nova_stream st;
  if (n != 7) return PyErr_Format(PyExc_TypeError, "seven arguments are needed");
  const nova_plan* plan = (const nova_plan*)PyLong_AsVoidPtr(a[0]);
  if (PyErr_Occurred()) return NULL;
  if (check(a[2], a[1]) != 1 || !shape(a[2], d, 4, 1) || !shape(a[3], u, 2, 0) || !pointer(a[2], &x) || !pointer(a[3], &U) ||
      !pointer(a[4], &y) || !pointer(a[5], &ws) || !integer(a[5], s_numel, &bytes))
    return NULL;
  const long flags = PyLong_AsLong(a[6]);
  if (PyErr_Occurred() || !stream(&st)) return NULL;
  int r;
  Py_BEGIN_ALLOW_THREADS
  r = fn.conv2d(plan, x, U, y, (int)d[0], (int)d[1], (int)d[2], (int)d[3], (int)u[1], ws, (size_t)bytes, (int)flags, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(r);
}

/* filter_transform(plan, g, K, C, U) -> status */
static PyObject* filter_transform(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *g, *U;
  nova_stream st;
  if (n != 5) return PyErr_Format(PyExc_TypeError, "five arguments are needed");
  const nova_plan* plan = (const nova_plan*)PyLong_AsVoidPtr(a[0]);
  const long K = PyLong_AsLong(a[2]), C = PyLong_AsLong(a[3]);
  if (PyErr_Occurred() || !pointer(a[1], &g) || !pointer(a[4], &U) || !stream(&st)) return NULL;
  int r;
  Py_BEGIN_ALLOW_THREADS
  r = fn.filter(plan, g, (int)K, (int)C, U, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(r);
}

/* conv2d_int8(plan, x, Uq, scale_U, scale_V, y, workspace, N, H, W, C, K, flags) -> status */
static PyObject* conv2d_int8(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *x, *U, *y, *ws, *sU;
  unsigned long long bytes;
  nova_stream st;
  long v[6];
  if (n != 13) return PyErr_Format(PyExc_TypeError, "thirteen arguments are needed");
  const nova_plan* plan = (const nova_plan*)PyLong_AsVoidPtr(a[0]);
  const double sV = PyFloat_AsDouble(a[4]);
  for (int i = 0; i < 6; ++i) v[i] = PyLong_AsLong(a[7 + i]);
  if (PyErr_Occurred() || !pointer(a[1], &x) || !pointer(a[2], &U) || !pointer(a[3], &sU) || !pointer(a[5], &y) ||
      !pointer(a[6], &ws) || !integer(a[6], s_numel, &bytes) || !stream(&st))
    return NULL;
  int r;
  Py_BEGIN_ALLOW_THREADS
  r = fn.int8(plan, x, U, (const float*)sU, (float)sV, y, (int)v[0], (int)v[1], (int)v[2], (int)v[3], (int)v[4], ws,
              (size_t)bytes, (int)v[5], st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(r);
}

/* bind(address of nova_conv2d_fwd, of nova_filter_transform, of nova_conv2d_fwd_int8, get_device, get_stream) */
static PyObject* bind(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  if (n != 5) return PyErr_Format(PyExc_TypeError, "five arguments are needed");
  *(void**)&fn.conv2d = PyLong_AsVoidPtr(a[0]);
  *(void**)&fn.filter = PyLong_AsVoidPtr(a[1]);
  *(void**)&fn.int8 = PyLong_AsVoidPtr(a[2]);
  if (PyErr_Occurred()) return NULL;
  Py_INCREF(a[3]);
  Py_INCREF(a[4]);
  Py_XSETREF(get_device, a[3]);
  Py_XSETREF(get_stream, a[4]);
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", (PyCFunction)(void (*)(void))bind, METH_FASTCALL, NULL},
    {"conv2d", (PyCFunction)(void (*)(void))conv2d, METH_FASTCALL, NULL},
    {"filter_transform", (PyCFunction)(void (*)(void))filter_transform, METH_FASTCALL, NULL},
    {"conv2d_int8", (PyCFunction)(void (*)(void))conv2d_int8, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_fastcall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fastcall(void) {
  s_is_cuda = PyUnicode_InternFromString("is_cuda");
  s_is_contiguous = PyUnicode_InternFromString("is_contiguous");
  s_dtype = PyUnicode_InternFromString("dtype");
  s_shape = PyUnicode_InternFromString("shape");
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_numel = PyUnicode_InternFromString("numel");
  return PyModule_Create(&module);
}
