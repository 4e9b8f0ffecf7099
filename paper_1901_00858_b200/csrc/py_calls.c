// CPython module `_calls`: the argument marshalling of the calls that a forward pass repeats.
//
// What bounds it: a program that runs layer by layer issues one call per layer, and small layers
// finish sooner than Python can issue the next one.  With ctypes a call of one launch cost about 8 us
// of host time, more than half of it conversions (3x3 layer, 3 -> 16 channels on 32x32: 11.4 -> 8.2 us
// a call; casting, folding and registering the weights of 49 layers, 147 calls: 1200 -> 642 us).  The
// functions convert the arguments (tensor -> address, stream -> handle), release the
// interpreter lock, call the C ABI through the addresses that bind() was given (of whichever
// build of the library the process has loaded) and return the hgc_status.
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

typedef int (*conv_fn)(void*, const void*, const void*, const void*, void*, int, void*);
typedef int (*dwpw_fn)(void*, const void*, const void*, const void*, const void*, const void*, void*, int, int, void*);
typedef int (*weights_fn)(void*, const void*, void*);
typedef int (*weights2_fn)(void*, const void*, const void*, void*);
typedef int (*cast_fn)(const void*, void*, int64_t, void*, void*);
typedef int (*fold_fn)(const void*, const void*, const void*, const void*, const void*, const void*, float, int32_t, int64_t, void*,
                       void*, void*);

static conv_fn f_forward, f_forward_host;
static dwpw_fn f_dwpw;
static weights_fn f_weights;
static weights2_fn f_weights2;
static cast_fn f_cast;
static fold_fn f_fold;

// torch's current device and its current stream on a device (set by stream_hooks; the callable
// given to bind() serves until then and sets them)
static PyObject *g_get_device, *g_get_stream, *g_first_stream;
static PyObject *s_data_ptr, *s_h, *s_value, *s_cuda_stream, *s_ctypes, *s_data, *s_numel, *s_size;
static PyObject* i_zero;

// Address of None (NULL), an int, a torch tensor or a numpy array.  0, or -1 with an exception set.
static int address(PyObject* t, void** out) {
  if (t == Py_None) {
    *out = NULL;
    return 0;
  }
  PyObject* v;
  if (PyLong_Check(t)) {
    v = Py_NewRef(t);
  } else {
    v = PyObject_CallMethodNoArgs(t, s_data_ptr);
    if (v == NULL && PyErr_ExceptionMatches(PyExc_AttributeError)) {
      PyErr_Clear();
      PyObject* c = PyObject_GetAttr(t, s_ctypes);
      if (c == NULL) return -1;
      v = PyObject_GetAttr(c, s_data);
      Py_DECREF(c);
    }
    if (v == NULL) return -1;
  }
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

// The stream handle of None (torch's current stream), an int or an object with .cuda_stream.
static int stream_handle(PyObject* s, void** out) {
  PyObject* v;
  if (s == Py_None) {
    if (g_get_stream != NULL) {
      PyObject* dev = PyObject_CallNoArgs(g_get_device);
      if (dev == NULL) return -1;
      v = PyObject_CallOneArg(g_get_stream, dev);
      Py_DECREF(dev);
    } else {
      v = PyObject_CallNoArgs(g_first_stream);
    }
  } else if (PyLong_Check(s)) {
    v = Py_NewRef(s);
  } else {
    v = PyObject_GetAttr(s, s_cuda_stream);
  }
  if (v == NULL) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

// The hgc_conv_desc* of a ConvDesc (its `_h` is a ctypes.c_void_p; NULL once it is closed).
static int desc_handle(PyObject* d, void** out) {
  PyObject* h = PyObject_GetAttr(d, s_h);
  if (h == NULL) return -1;
  PyObject* v = PyObject_GetAttr(h, s_value);
  Py_DECREF(h);
  if (v == NULL) return -1;
  const int rc = address(v, out);
  Py_DECREF(v);
  return rc;
}

static int count_is(Py_ssize_t n, Py_ssize_t want) {
  if (n == want) return 1;
  PyErr_Format(PyExc_TypeError, "%zd arguments, %zd are wanted", n, want);
  return 0;
}

// (desc, x, w, bias, y, relu, stream)
static PyObject* forward_with(conv_fn fn, PyObject* const* a, Py_ssize_t n) {
  void *d, *p[4], *st;
  if (!count_is(n, 7) || desc_handle(a[0], &d) < 0) return NULL;
  for (int i = 0; i < 4; ++i)
    if (address(a[1 + i], &p[i]) < 0) return NULL;
  const int relu = PyObject_IsTrue(a[5]);
  if (relu < 0 || stream_handle(a[6], &st) < 0) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = fn(d, p[0], p[1], p[2], p[3], relu, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static PyObject* conv_forward(PyObject* m, PyObject* const* a, Py_ssize_t n) { return forward_with(f_forward, a, n); }
static PyObject* conv_forward_host(PyObject* m, PyObject* const* a, Py_ssize_t n) { return forward_with(f_forward_host, a, n); }

// (desc, x, w_dw, bias_dw, w_pw, bias_pw, y, relu_dw, relu_pw, stream)
static PyObject* dwpw_forward(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  void *d, *p[6], *st;
  if (!count_is(n, 10) || desc_handle(a[0], &d) < 0) return NULL;
  for (int i = 0; i < 6; ++i)
    if (address(a[1 + i], &p[i]) < 0) return NULL;
  const int relu_dw = PyObject_IsTrue(a[7]), relu_pw = PyObject_IsTrue(a[8]);
  if (relu_dw < 0 || relu_pw < 0 || stream_handle(a[9], &st) < 0) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_dwpw(d, p[0], p[1], p[2], p[3], p[4], p[5], relu_dw, relu_pw, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (desc, w, stream) or, for blocks, (desc, w_dw, w_pw, stream)
static PyObject* set_weights(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  void *d, *w, *w2 = NULL, *st;
  if (n != 3 && !count_is(n, 4)) return NULL;
  if (desc_handle(a[0], &d) < 0 || address(a[1], &w) < 0 || (n == 4 && address(a[2], &w2) < 0) || stream_handle(a[n - 1], &st) < 0)
    return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = n == 3 ? f_weights(d, w, st) : f_weights2(d, w, w2, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

static int int_result(PyObject* v, int64_t* out) {
  if (v == NULL) return -1;
  *out = PyLong_AsLongLong(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

// (src, dst, count or None, overflow_count, stream)
static PyObject* cast_f32_to_f16(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  void *src, *dst, *over, *st;
  int64_t count;
  if (!count_is(n, 5) || address(a[0], &src) < 0 || address(a[1], &dst) < 0) return NULL;
  if (int_result(a[2] == Py_None ? PyObject_CallMethodNoArgs(a[0], s_numel) : Py_NewRef(a[2]), &count) < 0) return NULL;
  if (address(a[3], &over) < 0 || stream_handle(a[4], &st) < 0) return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_cast(src, dst, count, over, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (w, bias, mean, var, eps, w_out, b_out, gamma, beta, stream); k = w.size(0), per_k = w.numel() / k
static PyObject* bn_fold(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  static const int at[8] = {0, 1, 2, 3, 7, 8, 5, 6};  // w, bias, mean, var, gamma, beta, w_out, b_out
  void *p[8], *st;
  int64_t k, count;
  if (!count_is(n, 10)) return NULL;
  for (int i = 0; i < 8; ++i)
    if (address(a[at[i]], &p[i]) < 0) return NULL;
  const double eps = PyFloat_AsDouble(a[4]);
  if (eps == -1.0 && PyErr_Occurred()) return NULL;
  if (int_result(PyObject_CallMethodOneArg(a[0], s_size, i_zero), &k) < 0 ||
      int_result(PyObject_CallMethodNoArgs(a[0], s_numel), &count) < 0 || stream_handle(a[9], &st) < 0)
    return NULL;
  int rc;
  Py_BEGIN_ALLOW_THREADS
  rc = f_fold(p[0], p[1], p[2], p[3], p[4], p[5], (float)eps, (int32_t)k, k > 0 ? count / k : 0, p[6], p[7], st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(rc);
}

// (first_stream, forward, forward_host, dwpw_forward, set_weights, dwpw_set_weights, cast, bn_fold): the
// callable that finds torch's current stream the first time, and the functions' addresses
static PyObject* bind(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  void* p[7];
  if (!count_is(n, 8)) return NULL;
  for (int i = 0; i < 7; ++i)
    if (address(a[1 + i], &p[i]) < 0) return NULL;
  Py_XSETREF(g_first_stream, Py_NewRef(a[0]));
  f_forward = (conv_fn)p[0];
  f_forward_host = (conv_fn)p[1];
  f_dwpw = (dwpw_fn)p[2];
  f_weights = (weights_fn)p[3];
  f_weights2 = (weights2_fn)p[4];
  f_cast = (cast_fn)p[5];
  f_fold = (fold_fn)p[6];
  Py_RETURN_NONE;
}

// (current device, current stream handle of a device)
static PyObject* stream_hooks(PyObject* m, PyObject* const* a, Py_ssize_t n) {
  if (!count_is(n, 2)) return NULL;
  Py_XSETREF(g_get_device, Py_NewRef(a[0]));
  Py_XSETREF(g_get_stream, Py_NewRef(a[1]));
  Py_RETURN_NONE;
}

#define CALL(name) {#name, (PyCFunction)(void (*)(void))name, METH_FASTCALL, NULL}
static PyMethodDef methods[] = {CALL(conv_forward), CALL(conv_forward_host), CALL(dwpw_forward), CALL(set_weights),
                                CALL(cast_f32_to_f16), CALL(bn_fold), CALL(bind), CALL(stream_hooks), {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods};

PyMODINIT_FUNC PyInit__calls(void) {
  if ((s_data_ptr = PyUnicode_InternFromString("data_ptr")) == NULL || (s_h = PyUnicode_InternFromString("_h")) == NULL ||
      (s_value = PyUnicode_InternFromString("value")) == NULL || (s_cuda_stream = PyUnicode_InternFromString("cuda_stream")) == NULL ||
      (s_ctypes = PyUnicode_InternFromString("ctypes")) == NULL || (s_data = PyUnicode_InternFromString("data")) == NULL ||
      (s_numel = PyUnicode_InternFromString("numel")) == NULL || (s_size = PyUnicode_InternFromString("size")) == NULL ||
      (i_zero = PyLong_FromLong(0)) == NULL)
    return NULL;
  return PyModule_Create(&module);
}
