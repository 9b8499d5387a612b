/* CPython entry points of the calls that a program makes once per layer and pass
 * (wino_conv_forward, wino_conv_forward_static, wino_transform_weights,
 * wino_direct_conv_forward).  Argument marshalling only, as in binding.py, which keeps the
 * calls made once per plan.  The same marshalling through ctypes (argument objects, a stream
 * object, quantizer structs field by field) cost 8 to 10 us of host time a call, more than the
 * kernels of a small layer take; here it is a few hundred nanoseconds.
 *
 * A device address is a torch tensor (its data_ptr()), an int, or None.  A stream is None
 * (torch's current stream), an object with a `cuda_stream` attribute, or an int. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "wino.h"

static PyObject *s_data_ptr, *s_cuda_stream, *s_scale, *s_zero_point, *s_qmin, *s_qmax, *s_enabled;
static PyObject *get_device, *get_raw_stream; /* torch's accessors, resolved on first use */

/* Address behind `obj`; 0 on success, -1 with an exception set. */
static int address(PyObject *obj, void **out) {
  if (obj == Py_None) {
    *out = NULL;
    return 0;
  }
  PyObject *v = NULL;
  if (PyLong_Check(obj)) {
    *out = PyLong_AsVoidPtr(obj);
  } else {
    v = PyObject_CallMethodNoArgs(obj, s_data_ptr);
    if (v == NULL) return -1;
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
  }
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int current_stream(void **out) {
  if (get_raw_stream == NULL) {
    /* torch.cuda.current_stream() sets CUDA up if nothing has, or raises where there is none */
    PyObject *cuda = PyImport_ImportModule("torch.cuda");
    if (cuda == NULL) return -1;
    PyObject *s = PyObject_CallMethod(cuda, "current_stream", NULL);
    Py_DECREF(cuda);
    if (s == NULL) return -1;
    Py_DECREF(s);
    PyObject *c = PyImport_ImportModule("torch._C");
    if (c == NULL) return -1;
    PyObject *dev = PyObject_GetAttrString(c, "_cuda_getDevice");
    PyObject *raw = PyObject_GetAttrString(c, "_cuda_getCurrentRawStream");
    Py_DECREF(c);
    if (dev == NULL || raw == NULL) {
      Py_XDECREF(dev);
      Py_XDECREF(raw);
      return -1;
    }
    get_device = dev;
    get_raw_stream = raw;
  }
  PyObject *d = PyObject_CallNoArgs(get_device);
  if (d == NULL) return -1;
  PyObject *s = PyObject_CallOneArg(get_raw_stream, d);
  Py_DECREF(d);
  if (s == NULL) return -1;
  *out = PyLong_AsVoidPtr(s);
  Py_DECREF(s);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int stream_handle(PyObject *obj, void **out) {
  if (obj == Py_None) return current_stream(out);
  if (!PyLong_Check(obj)) {
    PyObject *v = PyObject_GetAttr(obj, s_cuda_stream);
    if (v == NULL) {
      PyErr_Clear();
      v = PyNumber_Long(obj);
      if (v == NULL) return -1;
    }
    *out = PyLong_AsVoidPtr(v);
    Py_DECREF(v);
  } else {
    *out = PyLong_AsVoidPtr(obj);
  }
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int as_int(PyObject *obj, int32_t *out) {
  PyObject *v = PyNumber_Long(obj); /* int(obj) */
  if (v == NULL) return -1;
  const long n = PyLong_AsLong(v);
  Py_DECREF(v);
  if (n == -1 && PyErr_Occurred()) return -1;
  if (n != (int32_t)n) {
    PyErr_SetString(PyExc_OverflowError, "value does not fit 32 bits");
    return -1;
  }
  *out = (int32_t)n;
  return 0;
}

/* Field of a dict or attribute of an object; NULL without an exception: not there. */
static PyObject *field(PyObject *q, PyObject *name) {
  if (PyDict_Check(q)) {
    PyObject *v = PyDict_GetItemWithError(q, name);
    Py_XINCREF(v);
    return v;
  }
  PyObject *v = PyObject_GetAttr(q, name);
  if (v == NULL && PyErr_ExceptionMatches(PyExc_AttributeError)) PyErr_Clear();
  return v;
}

static int quant_int(PyObject *q, PyObject *name, int32_t fallback, int32_t *out) {
  PyObject *v = field(q, name);
  if (v == NULL) {
    *out = fallback;
    return PyErr_Occurred() ? -1 : 0;
  }
  const int rc = as_int(v, out);
  Py_DECREF(v);
  return rc;
}

static int quant(PyObject *q, wino_quant_t *out) {
  PyObject *v = field(q, s_scale);
  if (v == NULL) {
    if (PyErr_Occurred()) return -1;
    out->scale = 1.0f;
  } else {
    const double d = PyFloat_AsDouble(v);
    Py_DECREF(v);
    if (d == -1.0 && PyErr_Occurred()) return -1;
    out->scale = (float)d;
  }
  if (quant_int(q, s_zero_point, 0, &out->zero_point) || quant_int(q, s_qmin, -127, &out->qmin) ||
      quant_int(q, s_qmax, 127, &out->qmax) || quant_int(q, s_enabled, 1, &out->enabled))
    return -1;
  return 0;
}

static int arg_count(const char *name, Py_ssize_t got, Py_ssize_t want) {
  if (got == want) return 0;
  PyErr_Format(PyExc_TypeError, "%s takes %zd arguments (%zd given)", name, want, got);
  return -1;
}

/* (plan, x, U_q, bias, y, workspace, stream) -> return code */
static PyObject *conv_forward(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  void *p[6], *st;
  if (arg_count("conv_forward", n, 7)) return NULL;
  for (int i = 0; i < 6; ++i)
    if (address(a[i], &p[i])) return NULL;
  if (stream_handle(a[6], &st)) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS /* a launch may wait for room in the queue */
  rc = wino_conv_forward(p[0], p[1], p[2], p[3], p[4], p[5], st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* (plan, x, U_q, bias, y, stream) -> return code */
static PyObject *conv_forward_static(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  void *p[5], *st;
  if (arg_count("conv_forward_static", n, 6)) return NULL;
  for (int i = 0; i < 5; ++i)
    if (address(a[i], &p[i])) return NULL;
  if (stream_handle(a[5], &st)) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS /* a launch may wait for room in the queue */
  rc = wino_conv_forward_static(p[0], p[1], p[2], p[3], p[4], st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* (plan, w, U_q, absmax, stream) -> return code */
static PyObject *transform_weights(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  void *p[4], *st;
  if (arg_count("transform_weights", n, 5)) return NULL;
  for (int i = 0; i < 4; ++i)
    if (address(a[i], &p[i])) return NULL;
  if (stream_handle(a[4], &st)) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS /* a launch may wait for room in the queue */
  rc = wino_transform_weights(p[0], p[1], p[2], p[3], st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

/* (N, C, H, W, K, stride, q_x, q_w, q_Y, x, w, bias, y, out_dtype, stream, s_w_K, s_Y_K) -> return code */
static PyObject *direct_conv_forward(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  wino_direct_desc_t d;
  void *p[4], *st, *s_w, *s_y;
  if (arg_count("direct_conv_forward", n, 17)) return NULL;
  int32_t *sizes[6] = {&d.N, &d.C, &d.H, &d.W, &d.K, &d.stride};
  for (int i = 0; i < 6; ++i)
    if (as_int(a[i], sizes[i])) return NULL;
  if (quant(a[6], &d.q_x) || quant(a[7], &d.q_w) || quant(a[8], &d.q_Y)) return NULL;
  for (int i = 0; i < 4; ++i)
    if (address(a[9 + i], &p[i])) return NULL;
  if (as_int(a[13], &d.out_dtype) || stream_handle(a[14], &st) || address(a[15], &s_w) ||
      address(a[16], &s_y))
    return NULL;
  d.s_w_K_dev = (const float *)s_w;
  d.s_Y_K_dev = (const float *)s_y;
  int rc;
  Py_BEGIN_ALLOW_THREADS /* a launch may wait for room in the queue */
  rc = wino_direct_conv_forward(&d, p[0], p[1], p[2], p[3], st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static PyMethodDef methods[] = {
    {"conv_forward", (PyCFunction)(void (*)(void))conv_forward, METH_FASTCALL, NULL},
    {"conv_forward_static", (PyCFunction)(void (*)(void))conv_forward_static, METH_FASTCALL, NULL},
    {"transform_weights", (PyCFunction)(void (*)(void))transform_weights, METH_FASTCALL, NULL},
    {"direct_conv_forward", (PyCFunction)(void (*)(void))direct_conv_forward, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_native", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__native(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  s_scale = PyUnicode_InternFromString("scale");
  s_zero_point = PyUnicode_InternFromString("zero_point");
  s_qmin = PyUnicode_InternFromString("qmin");
  s_qmax = PyUnicode_InternFromString("qmax");
  s_enabled = PyUnicode_InternFromString("enabled");
  if (!s_data_ptr || !s_cuda_stream || !s_scale || !s_zero_point || !s_qmin || !s_qmax || !s_enabled) return NULL;
  return PyModule_Create(&module);
}
