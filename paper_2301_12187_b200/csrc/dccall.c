/* The three forward calls of dc.py without ctypes: arguments are read from the Python objects here and the C entry point is
 * called through its address.  A small layer runs for 3-6 us, and marshalling its call through ctypes took 3.7 us of the host
 * (16 converted arguments, six pointers and the current stream fetched from Python); here about 1.
 *
 * Every function answers None for arguments that are not in the plain form it reads (a dtype it does not know, an act that
 * is no int, ...): dc.py then makes the call through ctypes, which reports what is wrong with them. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>

typedef int (*conv_fn)(const void *, int, int, int, const void *, const void *, const void *, int, const void *, void *, int,
                       void *, size_t, void *, int);
typedef int (*dw_fn)(const void *, int, int, int, int, int, int, int, const void *, const void *, int, void *, int, void *);
typedef int (*block_fn)(const void *, int, int, int, const void *, void *, int, void *, size_t, void *);

static conv_fn g_conv;
static dw_fn g_dw;
static block_fn g_block;
static PyObject *g_f32, *g_bf16, *g_geom, *g_block_type, *g_get_device, *g_get_stream;
static PyObject *s_data_ptr, *s_shape, *s_dtype, *s_numel, *s_element_size, *s_cuda_stream;

/* each reader: 0 on success, -1 when the argument has another form (any Python error is cleared by the caller) */
static int read_size(PyObject *o, size_t *v) {
  if (!o) return -1;
  const size_t r = PyLong_Check(o) ? PyLong_AsSize_t(o) : (size_t)-1;
  Py_DECREF(o);
  if (r == (size_t)-1) return -1;
  *v = r;
  return 0;
}
static int read_ptr(PyObject *t, void **p) {
  size_t v = 0;
  *p = NULL;
  if (t == Py_None) return 0;
  if (read_size(PyObject_CallMethodNoArgs(t, s_data_ptr), &v)) return -1;
  *p = (void *)v;
  return 0;
}
static int read_int(PyObject *o, int *v) {
  int overflow = 0;
  if (!PyLong_Check(o)) return -1;
  const long r = PyLong_AsLongAndOverflow(o, &overflow);
  if (overflow || r < -2147483647L - 1 || r > 2147483647L) return -1;
  *v = (int)r;
  return 0;
}
static int read_shape(PyObject *t, int *d) {
  PyObject *s = PyObject_GetAttr(t, s_shape);
  int bad = !s || !PyTuple_Check(s) || PyTuple_GET_SIZE(s) != 4;
  for (int i = 0; i < 4 && !bad; ++i) bad = read_int(PyTuple_GET_ITEM(s, i), &d[i]);
  Py_XDECREF(s);
  return bad ? -1 : 0;
}
static int read_dtype(PyObject *t, int *code) {
  PyObject *d = PyObject_GetAttr(t, s_dtype);
  Py_XDECREF(d);                                  /* dtypes are immortal singletons: compared, not used */
  if (d && d == g_f32) { *code = 0; return 0; }
  if (d && d == g_bf16) { *code = 1; return 0; }
  return -1;
}
static int read_bytes(PyObject *t, size_t *bytes) {
  size_t n = 0, e = 0;
  if (read_size(PyObject_CallMethodNoArgs(t, s_numel), &n) || read_size(PyObject_CallMethodNoArgs(t, s_element_size), &e)) return -1;
  *bytes = n * e;
  return 0;
}
static int read_stream(PyObject *stream, void **st) {
  size_t v = 0;
  if (stream == Py_None) {
    PyObject *dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return -1;
    PyObject *raw = PyObject_CallOneArg(g_get_stream, dev);
    Py_DECREF(dev);
    if (read_size(raw, &v)) return -1;
  } else if (read_size(PyObject_GetAttr(stream, s_cuda_stream), &v)) {
    return -1;
  }
  *st = (void *)v;
  return 0;
}
static PyObject *other_form(void) {
  PyErr_Clear();
  Py_RETURN_NONE;
}

/* conv(x, geom, w_packed, bias, act, residual, y, workspace, stream, algo) */
static PyObject *conv(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  int d[4], act, algo, code, st;
  void *x, *w, *b, *r, *y, *ws, *stream;
  size_t bytes;
  Py_buffer geom;
  if (n != 10 || !g_conv || (PyObject *)Py_TYPE(a[1]) != g_geom || read_shape(a[0], d) || read_dtype(a[0], &code) || read_ptr(a[0], &x) ||
      read_ptr(a[2], &w) || read_ptr(a[3], &b) || read_int(a[4], &act) || read_ptr(a[5], &r) || read_ptr(a[6], &y) ||
      read_ptr(a[7], &ws) || read_bytes(a[7], &bytes) || read_stream(a[8], &stream) || read_int(a[9], &algo) ||
      PyObject_GetBuffer(a[1], &geom, PyBUF_SIMPLE))
    return other_form();
  Py_BEGIN_ALLOW_THREADS
  st = g_conv(x, d[0], d[1], d[2], geom.buf, w, b, act, r, y, code, ws, bytes, stream, algo);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&geom);
  return PyLong_FromLong(st);
}

/* dwconv(x, k, stride, pad, w_packed, bias, act, y, stream) */
static PyObject *dwconv(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  int d[4], k, s, p, act, code, st;
  void *x, *w, *b, *y, *stream;
  if (n != 9 || !g_dw || read_shape(a[0], d) || read_dtype(a[0], &code) || read_ptr(a[0], &x) || read_int(a[1], &k) || read_int(a[2], &s) ||
      read_int(a[3], &p) || read_ptr(a[4], &w) || read_ptr(a[5], &b) || read_int(a[6], &act) || read_ptr(a[7], &y) ||
      read_stream(a[8], &stream))
    return other_form();
  Py_BEGIN_ALLOW_THREADS
  st = g_dw(x, d[0], d[1], d[2], d[3], k, s, p, w, b, act, y, code, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(st);
}

/* block(x, block, y, workspace, stream) */
static PyObject *block(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  int d[4], code, st;
  void *x, *y, *ws, *stream;
  size_t bytes;
  Py_buffer blk;
  if (n != 5 || !g_block || (PyObject *)Py_TYPE(a[1]) != g_block_type || read_shape(a[0], d) || read_dtype(a[0], &code) ||
      read_ptr(a[0], &x) || read_ptr(a[2], &y) || read_ptr(a[3], &ws) || read_bytes(a[3], &bytes) || read_stream(a[4], &stream) ||
      PyObject_GetBuffer(a[1], &blk, PyBUF_SIMPLE))
    return other_form();
  Py_BEGIN_ALLOW_THREADS
  st = g_block(x, d[0], d[1], d[2], blk.buf, y, code, ws, bytes, stream);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&blk);
  return PyLong_FromLong(st);
}

/* bind(conv address, dwconv address, block address, float32, bfloat16, Geom, Block, current device, current raw stream) */
static PyObject *bind(PyObject *self, PyObject *args) {
  unsigned long long c, w, b;
  PyObject *o[6];
  (void)self;
  if (!PyArg_ParseTuple(args, "KKKOOOOOO", &c, &w, &b, &o[0], &o[1], &o[2], &o[3], &o[4], &o[5])) return NULL;
  for (int i = 0; i < 6; ++i) Py_INCREF(o[i]);    /* kept for the life of the process */
  g_f32 = o[0]; g_bf16 = o[1]; g_geom = o[2]; g_block_type = o[3]; g_get_device = o[4]; g_get_stream = o[5];
  g_dw = (dw_fn)(uintptr_t)w;
  g_block = (block_fn)(uintptr_t)b;
  g_conv = (conv_fn)(uintptr_t)c;
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {{"conv", (PyCFunction)(void (*)(void))conv, METH_FASTCALL, NULL},
                                {"dwconv", (PyCFunction)(void (*)(void))dwconv, METH_FASTCALL, NULL},
                                {"block", (PyCFunction)(void (*)(void))block, METH_FASTCALL, NULL},
                                {"bind", bind, METH_VARARGS, NULL},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_dccall", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__dccall(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_shape = PyUnicode_InternFromString("shape");
  s_dtype = PyUnicode_InternFromString("dtype");
  s_numel = PyUnicode_InternFromString("numel");
  s_element_size = PyUnicode_InternFromString("element_size");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_data_ptr || !s_shape || !s_dtype || !s_numel || !s_element_size || !s_cuda_stream) return NULL;
  return PyModule_Create(&module);
}
