/*
 * fqt_py.c -- the argument marshalling of the Python binding in native code:
 * tensors and QTensor objects to the C ABI of include/fqt.h.
 *
 * A training step issues about five calls, and reading some sixty attributes
 * and data pointers from Python and through ctypes took 65 of the 97 us of a
 * small layer's step (128 x 256 x 256), more than its kernels.  Every call
 * reads the tensors as they are at that moment; nothing is kept between calls.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <string.h>

#include "fqt.h"

enum {
  A_CODES, A_CODES16, A_INV_S, A_ZERO, A_ROW_SUM, A_COL_SUM, A_LEAD, A_HZ, A_HR, A_PERM,
  A_GSTART, A_GSIZE, A_SHIFT16, A_SHIFT, A_SHIFT_COL_SUM, A_SHIFT_SCALE, A_POINTERS,
  A_BITS = A_POINTERS, A_KIND, A_BLOCK, A_ROWS_PER_SAMPLE, A_CONV, A_LOGICAL, A_SHAPE,
  A_DATA_PTR, A_COUNT
};
static const char *const kNames[A_COUNT] = {
    "codes", "codes16", "inv_s", "zero", "row_sum", "col_sum", "lead", "hz", "hr", "perm",
    "gstart", "gsize", "shift16", "shift", "shift_col_sum", "shift_scale", "bits", "kind",
    "block", "rows_per_sample", "conv", "logical", "shape", "data_ptr"};
static PyObject *g_name[A_COUNT];

/* data_ptr() of a tensor; -1 with an exception set on failure (AttributeError
 * for None) */
static int needed_ptr(PyObject *t, void **out) {
  *out = NULL;
  PyObject *v = PyObject_CallMethodNoArgs(t, g_name[A_DATA_PTR]);
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

/* the same with 0 for None */
static int tensor_ptr(PyObject *t, void **out) {
  *out = NULL;
  return t == Py_None ? 0 : needed_ptr(t, out);
}

static int int_attr(PyObject *o, int name, int32_t *out) {
  PyObject *v = PyObject_GetAttr(o, g_name[name]);
  if (!v) return -1;
  *out = (int32_t)PyLong_AsLong(v);
  Py_DECREF(v);
  return PyErr_Occurred() ? -1 : 0;
}

/* the entries of a sequence of two integers */
static int two_ints(PyObject *seq, int64_t *a, int64_t *b) {
  PyObject *f = PySequence_Fast(seq, "shape");
  if (!f) return -1;
  if (PySequence_Fast_GET_SIZE(f) == 2) {
    *a = PyLong_AsLongLong(PySequence_Fast_GET_ITEM(f, 0));
    *b = PyLong_AsLongLong(PySequence_Fast_GET_ITEM(f, 1));
  } else {
    PyErr_Format(PyExc_ValueError, "a quantized tensor has two dimensions, not %zd",
                 PySequence_Fast_GET_SIZE(f));
  }
  Py_DECREF(f);
  return PyErr_Occurred() ? -1 : 0;
}

/* A QTensor object as the C struct (AttributeError for None). */
static int fill(PyObject *q, fqt_qtensor *s, fqt_qtensor **out) {
  *out = NULL;
  memset(s, 0, sizeof(*s));
  void *p[A_POINTERS];
  PyObject *matrix = NULL; /* the codes whose shape is the tensor's */
  int bad = 0;
  for (int i = 0; i < A_POINTERS && !bad; ++i) {
    PyObject *t = PyObject_GetAttr(q, g_name[i]);
    if (!t) { bad = 1; break; }
    bad = (i == A_INV_S || i == A_ZERO ? needed_ptr(t, &p[i]) : tensor_ptr(t, &p[i])) != 0;
    if (!matrix && i <= A_CODES16 && t != Py_None) matrix = t;  /* keeps the reference */
    else Py_DECREF(t);
  }
  if (!bad) {
    PyObject *logical = PyObject_GetAttr(q, g_name[A_LOGICAL]);
    PyObject *shape = NULL;
    if (!logical) bad = 1;
    else if (logical != Py_None) shape = Py_NewRef(logical);
    else if (matrix) shape = PyObject_GetAttr(matrix, g_name[A_SHAPE]);
    else PyErr_SetString(PyExc_AttributeError, "a quantized tensor needs codes or codes16");
    Py_XDECREF(logical);
    bad = bad || !shape || two_ints(shape, &s->rows, &s->cols) != 0;
    Py_XDECREF(shape);
  }
  Py_XDECREF(matrix);
  if (bad || int_attr(q, A_BITS, &s->bits) || int_attr(q, A_KIND, &s->kind) ||
      int_attr(q, A_BLOCK, &s->block) || int_attr(q, A_ROWS_PER_SAMPLE, &s->rows_per_sample))
    return -1;
  PyObject *conv = PyObject_GetAttr(q, g_name[A_CONV]);
  if (!conv) return -1;
  const int given = PyObject_IsTrue(conv); /* None or empty: not a conv operand */
  PyObject *f = given > 0 ? PySequence_Fast(conv, "conv") : NULL;
  if (f && PySequence_Fast_GET_SIZE(f) <= 8) {
    for (Py_ssize_t i = 0; i < PySequence_Fast_GET_SIZE(f) && !PyErr_Occurred(); ++i)
      s->conv[i] = (int32_t)PyLong_AsLong(PySequence_Fast_GET_ITEM(f, i));
  } else if (f) {
    PyErr_SetString(PyExc_IndexError, "conv holds eight integers");
  }
  Py_XDECREF(f);
  Py_DECREF(conv);
  if (PyErr_Occurred()) return -1;
  s->codes = p[A_CODES];
  s->codes_f16 = p[A_CODES16];
  s->inv_s = p[A_INV_S];
  s->zero = p[A_ZERO];
  s->row_sum = p[A_ROW_SUM];
  s->col_sum = p[A_COL_SUM];
  s->lead = p[A_LEAD];
  s->hz = p[A_HZ];
  s->hr = p[A_HR];
  s->perm = p[A_PERM];
  s->gstart = p[A_GSTART];
  s->gsize = p[A_GSIZE];
  s->shift_f16 = p[A_SHIFT16];
  s->shift = p[A_SHIFT];
  s->shift_col_sum = p[A_SHIFT_COL_SUM];
  s->shift_scale = p[A_SHIFT_SCALE];
  *out = s;
  return 0;
}

/* The same for an operand that may be left out: NULL for None. */
static int fill_optional(PyObject *q, fqt_qtensor *s, fqt_qtensor **out) {
  *out = NULL;
  return q == Py_None ? 0 : fill(q, s, out);
}

#define NARGS(k)                                                     \
  if (n != (k)) {                                                    \
    PyErr_SetString(PyExc_TypeError, "wrong number of arguments");   \
    return NULL;                                                     \
  }
#define I64(i) PyLong_AsLongLong(a[i])
#define INT(i) ((int)PyLong_AsLong(a[i]))

/* a call of the C ABI, without the interpreter lock; its status is the result */
#define CALL(expr)                \
  fqt_status st_;                 \
  Py_BEGIN_ALLOW_THREADS          \
  st_ = (expr);                   \
  Py_END_ALLOW_THREADS            \
  return PyLong_FromLong(st_);

/* the last three arguments of every call: workspace tensor, bytes, stream */
typedef struct {
  void *ws, *stream;
  size_t bytes;
} Tail;

static int tail(PyObject *const *a, Tail *t) {
  if (needed_ptr(a[0], &t->ws)) return -1;
  t->bytes = PyLong_AsSize_t(a[1]);
  t->stream = PyLong_AsVoidPtr(a[2]);
  return PyErr_Occurred() ? -1 : 0;
}

/* quantize_fwd(weight, X, dtype, rows, cols, bits, out, ws, bytes, stream) */
static PyObject *py_quantize_fwd(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  NARGS(10)
  void *x;
  fqt_qtensor s, *q;
  Tail t;
  const int weight = INT(0);
  const fqt_dtype dt = (fqt_dtype)INT(2);
  const int64_t rows = I64(3), cols = I64(4);
  const int bits = INT(5);
  if (PyErr_Occurred() || tensor_ptr(a[1], &x) || fill(a[6], &s, &q) || tail(a + 7, &t))
    return NULL;
  CALL(weight ? fqt_quantize_weight(x, dt, rows, cols, bits, q, t.ws, t.bytes, t.stream)
              : fqt_quantize_act(x, dt, rows, cols, bits, q, t.ws, t.bytes, t.stream))
}

/* quantize_act_conv(X, dtype, n, h, w, c, kh, kw, pad, bits, out, ws, bytes, stream) */
static PyObject *py_quantize_act_conv(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  NARGS(14)
  void *x;
  fqt_qtensor s, *q;
  Tail t;
  const fqt_dtype dt = (fqt_dtype)INT(1);
  const int64_t im = I64(2), h = I64(3), w = I64(4), c = I64(5);
  const int kh = INT(6), kw = INT(7), pad = INT(8), bits = INT(9);
  if (PyErr_Occurred() || tensor_ptr(a[0], &x) || fill(a[10], &s, &q) || tail(a + 11, &t))
    return NULL;
  CALL(fqt_quantize_act_conv(x, dt, im, h, w, c, kh, kw, pad, bits, q, t.ws, t.bytes, t.stream))
}

/* quantize_grad_samples(dH, dtype, N, C, R, kind, bits, seed, q_b2, q_b1, ws, bytes, stream) */
static PyObject *py_quantize_grad_samples(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  NARGS(13)
  void *h;
  fqt_qtensor s2, s1, *q2, *q1;
  Tail t;
  const fqt_dtype dt = (fqt_dtype)INT(1);
  const int64_t N = I64(2), C = I64(3), R = I64(4);
  const fqt_kind kind = (fqt_kind)INT(5);
  const int bits = INT(6);
  const uint64_t seed = PyLong_AsUnsignedLongLong(a[7]);
  if (PyErr_Occurred() || tensor_ptr(a[0], &h) || fill(a[8], &s2, &q2) ||
      fill_optional(a[9], &s1, &q1) || tail(a + 10, &t))
    return NULL;
  CALL(fqt_quantize_grad_samples(h, dt, N, C, R, kind, bits, seed, q2, q1, t.ws, t.bytes,
                                 t.stream))
}

/* conv_grad_x_nhwc(q_b2, qw, n, h, w, cin, k, pad, grad_X, ws, bytes, stream) */
static PyObject *py_conv_grad_x_nhwc(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  NARGS(12)
  fqt_qtensor s[2], *q[2];
  void *gx;
  Tail t;
  const int64_t im = I64(2), h = I64(3), w = I64(4), cin = I64(5);
  const int k = INT(6), pad = INT(7);
  if (PyErr_Occurred() || fill(a[0], &s[0], &q[0]) || fill(a[1], &s[1], &q[1]) ||
      tensor_ptr(a[8], &gx) || tail(a + 9, &t))
    return NULL;
  CALL(fqt_conv_grad_x_nhwc(q[0], q[1], im, h, w, cin, k, pad, gx, t.ws, t.bytes, t.stream))
}

/* quantize_grad(dH, dtype, N, C, kind, bits, block, seed, q_b2, q_b1, ws, bytes, stream) */
static PyObject *py_quantize_grad(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  NARGS(13)
  void *h;
  fqt_qtensor s2, s1, *q2, *q1;
  Tail t;
  const fqt_dtype dt = (fqt_dtype)INT(1);
  const int64_t N = I64(2), C = I64(3);
  const fqt_kind kind = (fqt_kind)INT(4);
  const int bits = INT(5), block = INT(6);
  const uint64_t seed = PyLong_AsUnsignedLongLong(a[7]);
  if (PyErr_Occurred() || tensor_ptr(a[0], &h) || fill(a[8], &s2, &q2) ||
      fill_optional(a[9], &s1, &q1) || tail(a + 10, &t))
    return NULL;
  CALL(fqt_quantize_grad(h, dt, N, C, kind, bits, block, seed, q2, q1, t.ws, t.bytes, t.stream))
}

/* linear_backward(q_b2, q_b1, qx, qw, grad_X, grad_W, ws, bytes, stream) */
static PyObject *py_linear_backward(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  NARGS(9)
  fqt_qtensor s[4], *q[4];
  void *gx, *gw;
  Tail t;
  if (fill(a[0], &s[0], &q[0])) return NULL;
  for (int i = 1; i < 4; ++i)
    if (fill_optional(a[i], &s[i], &q[i])) return NULL;
  if (tensor_ptr(a[4], &gx) || tensor_ptr(a[5], &gw) || tail(a + 6, &t)) return NULL;
  CALL(fqt_linear_backward(q[0], q[1], q[2], q[3], gx, gw, t.ws, t.bytes, t.stream))
}

/* linear_forward(qx, qw, H, ws, bytes, stream) */
static PyObject *py_linear_forward(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  NARGS(6)
  fqt_qtensor s[2], *q[2];
  void *h;
  Tail t;
  if (fill(a[0], &s[0], &q[0]) || fill(a[1], &s[1], &q[1]) || tensor_ptr(a[2], &h) ||
      tail(a + 3, &t))
    return NULL;
  CALL(fqt_linear_forward(q[0], q[1], h, t.ws, t.bytes, t.stream))
}

/* workspace_size(N, C, D) */
static PyObject *py_workspace_size(PyObject *self, PyObject *const *a, Py_ssize_t n) {
  (void)self;
  NARGS(3)
  const int64_t N = I64(0), C = I64(1), D = I64(2);
  if (PyErr_Occurred()) return NULL;
  return PyLong_FromSize_t(fqt_workspace_size(N, C, D));
}

static PyMethodDef kMethods[] = {
    {"quantize_fwd", (PyCFunction)(void (*)(void))py_quantize_fwd, METH_FASTCALL, NULL},
    {"quantize_act_conv", (PyCFunction)(void (*)(void))py_quantize_act_conv, METH_FASTCALL, NULL},
    {"quantize_grad_samples", (PyCFunction)(void (*)(void))py_quantize_grad_samples,
     METH_FASTCALL, NULL},
    {"conv_grad_x_nhwc", (PyCFunction)(void (*)(void))py_conv_grad_x_nhwc, METH_FASTCALL, NULL},
    {"quantize_grad", (PyCFunction)(void (*)(void))py_quantize_grad, METH_FASTCALL, NULL},
    {"linear_backward", (PyCFunction)(void (*)(void))py_linear_backward, METH_FASTCALL, NULL},
    {"linear_forward", (PyCFunction)(void (*)(void))py_linear_forward, METH_FASTCALL, NULL},
    {"workspace_size", (PyCFunction)(void (*)(void))py_workspace_size, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "_fqt_py", NULL, -1, kMethods,
                                     NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__fqt_py(void) {
  for (int i = 0; i < A_COUNT; ++i)
    if (!(g_name[i] = PyUnicode_InternFromString(kNames[i]))) return NULL;
  return PyModule_Create(&kModule);
}
