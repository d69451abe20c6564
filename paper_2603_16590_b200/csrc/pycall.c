/* CPython shim for the calls a program makes per layer and step: takes the tensors themselves, reads what the
 * C entry point wants to know of them and calls it.  Through ctypes the same marshalling (eleven arguments
 * converted one by one, as many attribute look-ups from bytecode) took 3.6 us of a call's 8.5.
 * No arithmetic, no checks of its own: those are the library's. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

static PyObject *s_data_ptr, *s_size, *s_shape, *s_stride, *s_numel, *s_dtype, *zero, *one, *float32_type;
static PyTypeObject *tensor_type;

typedef int (*linear_fn)(const void *, const void *, const void *, int64_t, int64_t, void *, int32_t, int64_t, void *, size_t,
                         void *);
typedef int (*quantise_fn)(const void *, const void *, int64_t, int64_t, int64_t, void *, void *, int32_t, void *);

/* A tensor's data pointer, None, or whatever int() takes; bits above 64 are dropped, as ctypes does. */
static int as_pointer(PyObject *o, void **out) {
  if (o == Py_None) { *out = NULL; return 0; }
  PyObject *r = PyLong_Check(o)                        ? Py_NewRef(o)
                : PyObject_TypeCheck(o, tensor_type) ? PyObject_CallMethodNoArgs(o, s_data_ptr)
                                                     : PyNumber_Long(o);
  if (r == NULL) return -1;
  *out = (void *)(uintptr_t)PyLong_AsUnsignedLongLongMask(r);
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

/* x.shape[i]; of a tensor without the torch.Size. */
static int as_extent(PyObject *o, PyObject *i, int64_t *out) {
  if (PyObject_TypeCheck(o, tensor_type)) return as_int(o, s_size, i, out);
  PyObject *shape = PyObject_GetAttr(o, s_shape);
  if (shape == NULL) return -1;
  PyObject *r = PyObject_GetItem(shape, i);
  Py_DECREF(shape);
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
  if (as_pointer(a[0], &fn) || as_pointer(a[1], &t) || as_pointer(a[2], &w) || as_extent(a[3], zero, &s) ||
      as_int(a[3], s_stride, zero, &ld) || as_pointer(a[3], &x) || as_pointer(a[4], &y) ||
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
  if (as_pointer(a[0], &fn) || as_pointer(a[1], &t) || as_extent(a[2], zero, &s) || as_extent(a[2], one, &cols) ||
      as_int(a[2], s_stride, zero, &ld) || as_pointer(a[2], &x) || as_pointer(a[3], &codes) ||
      as_pointer(a[4], &scales) || as_pointer(a[6], &stream))
    return NULL;
  if (!PyLong_Check(a[5])) { PyErr_SetString(PyExc_TypeError, "quantise: scale_layout is not an int"); return NULL; }
  const unsigned long layout = PyLong_AsUnsignedLongMask(a[5]);
  int st;
  Py_BEGIN_ALLOW_THREADS
  st = ((quantise_fn)fn)(t, x, s, cols, ld, codes, scales, (int32_t)layout, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

/* setup(torch.float32, torch.Tensor) */
static PyObject *setup(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  if (n != 2 || !PyType_Check(a[1])) { PyErr_SetString(PyExc_TypeError, "setup: a dtype and a type"); return NULL; }
  Py_XSETREF(float32_type, Py_NewRef(a[0]));
  Py_XSETREF(tensor_type, (PyTypeObject *)Py_NewRef(a[1]));
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"linear", (PyCFunction)(void (*)(void))linear, METH_FASTCALL, NULL},
                                {"quantise", (PyCFunction)(void (*)(void))quantise, METH_FASTCALL, NULL},
                                {"setup", (PyCFunction)(void (*)(void))setup, METH_FASTCALL, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_pycall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__pycall(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_size = PyUnicode_InternFromString("size");
  s_shape = PyUnicode_InternFromString("shape");
  s_stride = PyUnicode_InternFromString("stride");
  s_numel = PyUnicode_InternFromString("numel");
  s_dtype = PyUnicode_InternFromString("dtype");
  zero = PyLong_FromLong(0);
  one = PyLong_FromLong(1);
  if (!s_data_ptr || !s_size || !s_shape || !s_stride || !s_numel || !s_dtype || !zero || !one) return NULL;
  return PyModule_Create(&module);
}
