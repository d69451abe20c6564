/* CPython shim for the calls a program makes per layer and step: takes the tensors themselves, reads what the
 * C entry point wants to know of them and calls it.  Through ctypes the same marshalling (eleven arguments
 * converted one by one, as many attribute look-ups from bytecode) took 3.6 us of a call's 8.5.
 * No arithmetic, no checks of its own: those are the library's. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

static PyObject *s_data_ptr, *s_size, *s_stride, *s_numel, *s_dtype, *zero, *one, *float32_type;

typedef int (*linear_fn)(const void *, const void *, const void *, int64_t, int64_t, void *, int32_t, int64_t, void *, size_t,
                         void *);
typedef int (*quantise_fn)(const void *, const void *, int64_t, int64_t, int64_t, void *, void *, int32_t, void *);

/* A tensor's data pointer, a plain integer, or None. */
static int as_pointer(PyObject *o, void **out) {
  if (o == Py_None) { *out = NULL; return 0; }
  if (PyLong_Check(o)) {
    *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLong(o);
    return PyErr_Occurred() ? -1 : 0;
  }
  PyObject *r = PyObject_CallMethodNoArgs(o, s_data_ptr);
  if (r == NULL) return -1;
  *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLong(r);
  Py_DECREF(r);
  return PyErr_Occurred() ? -1 : 0;
}

static int as_int(PyObject *o, PyObject *method, PyObject *arg, int64_t *out) {
  PyObject *r = arg ? PyObject_CallMethodOneArg(o, method, arg) : PyObject_CallMethodNoArgs(o, method);
  if (r == NULL) return -1;
  *out = (int64_t)PyLong_AsLongLong(r);
  Py_DECREF(r);
  return PyErr_Occurred() ? -1 : 0;
}

/* linear(function, transform, weight, x, y, workspace, stream) -> status */
static PyObject *linear(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  if (n != 7) { PyErr_SetString(PyExc_TypeError, "linear: 7 arguments"); return NULL; }
  void *fn, *t, *w, *x, *y, *ws, *stream;
  int64_t s, ld, ldy, bytes;
  if (as_pointer(a[0], &fn) || as_pointer(a[1], &t) || as_pointer(a[2], &w) || as_pointer(a[3], &x) ||
      as_int(a[3], s_size, zero, &s) || as_int(a[3], s_stride, zero, &ld) || as_pointer(a[4], &y) ||
      as_int(a[4], s_stride, zero, &ldy) || as_pointer(a[5], &ws) || as_int(a[5], s_numel, NULL, &bytes) ||
      as_pointer(a[6], &stream))
    return NULL;
  PyObject *dt = PyObject_GetAttr(a[4], s_dtype);
  if (dt == NULL) return NULL;
  const int32_t y_dtype = dt == float32_type ? 0 : 1;   /* BATQ_F32, BATQ_BF16 */
  Py_DECREF(dt);
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = ((linear_fn)fn)(t, w, x, s, ld, y, y_dtype, ldy, ws, (size_t)bytes, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

/* quantise(function, transform, x, codes, scales, scale_layout, stream) -> status */
static PyObject *quantise(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  if (n != 7) { PyErr_SetString(PyExc_TypeError, "quantise: 7 arguments"); return NULL; }
  void *fn, *t, *x, *codes, *scales, *stream;
  int64_t s, cols, ld;
  if (as_pointer(a[0], &fn) || as_pointer(a[1], &t) || as_pointer(a[2], &x) || as_int(a[2], s_size, zero, &s) ||
      as_int(a[2], s_size, one, &cols) || as_int(a[2], s_stride, zero, &ld) || as_pointer(a[3], &codes) ||
      as_pointer(a[4], &scales) || as_pointer(a[6], &stream))
    return NULL;
  const long layout = PyLong_AsLong(a[5]);
  if (layout == -1 && PyErr_Occurred()) return NULL;
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = ((quantise_fn)fn)(t, x, s, cols, ld, codes, scales, (int32_t)layout, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

/* setup(torch.float32) */
static PyObject *setup(PyObject *self, PyObject *dtype) {
  (void)self;
  Py_INCREF(dtype);
  Py_XSETREF(float32_type, dtype);
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"linear", (PyCFunction)(void (*)(void))linear, METH_FASTCALL, NULL},
                                {"quantise", (PyCFunction)(void (*)(void))quantise, METH_FASTCALL, NULL},
                                {"setup", setup, METH_O, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_size = PyUnicode_InternFromString("size");
  s_stride = PyUnicode_InternFromString("stride");
  s_numel = PyUnicode_InternFromString("numel");
  s_dtype = PyUnicode_InternFromString("dtype");
  zero = PyLong_FromLong(0);
  one = PyLong_FromLong(1);
  if (!s_data_ptr || !s_size || !s_stride || !s_numel || !s_dtype || !zero || !one) return NULL;
  return PyModule_Create(&module);
}
