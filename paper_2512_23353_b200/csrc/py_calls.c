/* Native argument marshalling for the calls of a layer's pass: what binding.py does with ctypes, in a third of the time (a pass
 * over a small layer is bound by the host: ctypes and the checks were 8 of its 25 us).
 *
 * Every function checks its tensors as binding.py does and calls the library with the interpreter lock released.  It returns the
 * library's status, or None if anything is not as expected (an offsets list, a wrong dtype or size, a failing attribute):
 * binding.py then goes through its own checks, which convert the argument or raise. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "isopo.h"

static struct {
  isopo_status (*layer_gram)(const void*, const void*, isopo_dtype, int64_t, int, int, const int64_t*, int, isopo_path, float*,
                             void*, size_t, int32_t*, void*);
  isopo_status (*transform)(const float*, const float*, int, isopo_variant, float, const float*, float*, int32_t*, void*);
  isopo_status (*transform_rel)(const float*, const float*, int, isopo_variant, float, const float*, const float*, float*,
                                int32_t*, void*);
  isopo_status (*reg_ema)(const float*, int, float, float*, void*);
  isopo_status (*weight_grad)(const void*, const void*, isopo_dtype, int64_t, int, int, const float*, const int64_t*, int,
                              isopo_path, float*, float, void*, size_t, int32_t*, void*);
  isopo_status (*sampled)(const void*, const void*, isopo_dtype, int64_t, int, int, const int64_t*, int, const int64_t*, int,
                          const float*, float, float*, float*, void*, size_t, int32_t*, void*);
} lib;
static PyObject *dt_f32, *dt_bf16, *dt_i32, *dt_u8, *get_device, *get_stream;
static PyObject *s_data_ptr, *s_dtype, *s_is_cuda, *s_is_contiguous, *s_numel, *s_shape;

/* All helpers return 0 on success; a failure may leave an exception set, which `giving_up` clears. */
static PyObject* giving_up(void) {
  PyErr_Clear();
  Py_RETURN_NONE;
}
static int call_int(PyObject* t, PyObject* method, long long* out) {
  PyObject* r = PyObject_VectorcallMethod(method, &t, 1, NULL);
  if (!r) return -1;
  *out = PyLong_AsLongLong(r);
  Py_DECREF(r);
  return *out == -1 && PyErr_Occurred() ? -1 : 0;
}
static int is_true(PyObject* r) { /* steals r */
  const int yes = r == Py_True;
  Py_XDECREF(r);
  return yes;
}
static int has_dtype(PyObject* t, PyObject* dtype) {
  PyObject* r = PyObject_GetAttr(t, s_dtype);
  Py_XDECREF(r);
  return r == dtype;
}
static int address(PyObject* t, void** p) {
  long long v;
  if (call_int(t, s_data_ptr, &v)) return -1;
  *p = (void*)(uintptr_t)v;
  return 0;
}
static int contiguous(PyObject* t) {
  return is_true(PyObject_VectorcallMethod(s_is_contiguous, &t, 1, NULL));
}
static int on_cuda(PyObject* t) { return is_true(PyObject_GetAttr(t, s_is_cuda)); }
/* a tensor of `dtype` and n elements (any number: n < 0) */
static int vector(PyObject* t, PyObject* dtype, long long n, void** p) {
  long long have;
  if (!has_dtype(t, dtype)) return -1;
  if (n >= 0 && (call_int(t, s_numel, &have) || have != n)) return -1;
  return address(t, p);
}
static int matrix_shape(PyObject* t, long long* rows, long long* cols) {
  PyObject* s = PyObject_GetAttr(t, s_shape);
  if (!s) return -1;
  const int ok = PyTuple_Check(s) && PyTuple_GET_SIZE(s) == 2;
  if (ok) {
    *rows = PyLong_AsLongLong(PyTuple_GET_ITEM(s, 0));
    *cols = PyLong_AsLongLong(PyTuple_GET_ITEM(s, 1));
  }
  Py_DECREF(s);
  return ok && *rows >= 0 && *cols >= 0 && *rows <= INT32_MAX && *cols <= INT32_MAX ? 0 : -1;
}
/* X and dY: same dtype, shapes */
typedef struct { void *X, *dY; isopo_dtype dtype; long long T, d_in, d_out; } Operands;
static int operands(PyObject* X, PyObject* dY, int check_layout, Operands* o) {
  long long rows;
  if (has_dtype(X, dt_bf16)) o->dtype = ISOPO_BF16;
  else if (has_dtype(X, dt_f32)) o->dtype = ISOPO_F32;
  else return -1;
  if (check_layout && (!has_dtype(dY, o->dtype == ISOPO_BF16 ? dt_bf16 : dt_f32) || !on_cuda(X) || !on_cuda(dY) ||
                       !contiguous(X) || !contiguous(dY)))
    return -1;
  if (matrix_shape(X, &o->T, &o->d_in) || matrix_shape(dY, &rows, &o->d_out)) return -1;
  return address(X, &o->X) || address(dY, &o->dY) ? -1 : 0;
}
/* int64 values in one contiguous row */
static int int64_row(PyObject* a, Py_buffer* view) {
  if (PyObject_GetBuffer(a, view, PyBUF_FORMAT | PyBUF_C_CONTIGUOUS)) return -1;
  if (view->ndim == 1 && view->itemsize == 8 && view->format && view->format[0] == 'l' && view->format[1] == 0 &&
      view->shape[0] >= 2 && view->shape[0] <= INT32_MAX)
    return 0;
  PyBuffer_Release(view);
  return -1;
}
/* B + 1 offsets */
static int offsets(PyObject* a, Py_buffer* view, int* B) {
  if (int64_row(a, view)) return -1;
  *B = (int)view->shape[0] - 1;
  return 0;
}
static int stream(void** st) {
  PyObject* dev = PyObject_CallNoArgs(get_device);
  if (!dev) return -1;
  PyObject* r = PyObject_CallOneArg(get_stream, dev);
  Py_DECREF(dev);
  if (!r) return -1;
  *st = PyLong_AsVoidPtr(r);
  Py_DECREF(r);
  return PyErr_Occurred() ? -1 : 0;
}
static int int_arg(PyObject* a, int* v) {
  if (!PyLong_CheckExact(a)) return -1;
  const long x = PyLong_AsLong(a);
  if (x < 0 || x > INT32_MAX) return -1;
  *v = (int)x;
  return 0;
}
static int float_arg(PyObject* a, float* v) {
  if (!PyFloat_Check(a)) return -1;
  *v = (float)PyFloat_AS_DOUBLE(a);
  return 0;
}

/* layer_gram(X, dY, offsets, K, ws, info, path) */
static PyObject* layer_gram(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Operands o;
  Py_buffer off;
  void *K, *ws, *info, *st;
  long long ws_bytes;
  int B, path;
  if (n != 7 || offsets(a[2], &off, &B)) return giving_up();
  if (operands(a[0], a[1], 1, &o) || !contiguous(a[3]) || vector(a[3], dt_f32, (long long)B * B, &K) ||
      vector(a[4], dt_u8, -1, &ws) || call_int(a[4], s_numel, &ws_bytes) || vector(a[5], dt_i32, -1, &info) ||
      int_arg(a[6], &path) || stream(&st)) {
    PyBuffer_Release(&off);
    return giving_up();
  }
  isopo_status s;
  Py_BEGIN_ALLOW_THREADS
  s = lib.layer_gram(o.X, o.dY, o.dtype, o.T, (int)o.d_in, (int)o.d_out, (const int64_t*)off.buf, B, (isopo_path)path, (float*)K,
                     ws, (size_t)ws_bytes, (int32_t*)info, st);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&off);
  return PyLong_FromLong(s);
}

/* weight_grad(X, dY, coeffs, offsets, dW, ws, info, path, beta) */
static PyObject* weight_grad(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Operands o;
  Py_buffer off;
  void *c, *dW, *ws, *info, *st;
  long long ws_bytes, rows, cols;
  int B, path;
  float beta;
  if (n != 9 || offsets(a[3], &off, &B)) return giving_up();
  if (operands(a[0], a[1], 0, &o) || vector(a[2], dt_f32, B, &c) || vector(a[4], dt_f32, -1, &dW) || !contiguous(a[4]) ||
      matrix_shape(a[4], &rows, &cols) || rows != o.d_out || cols != o.d_in || address(a[5], &ws) ||
      call_int(a[5], s_numel, &ws_bytes) || address(a[6], &info) || int_arg(a[7], &path) || float_arg(a[8], &beta) ||
      stream(&st)) {
    PyBuffer_Release(&off);
    return giving_up();
  }
  isopo_status s;
  Py_BEGIN_ALLOW_THREADS
  s = lib.weight_grad(o.X, o.dY, o.dtype, o.T, (int)o.d_in, (int)o.d_out, (const float*)c, (const int64_t*)off.buf, B,
                      (isopo_path)path, (float*)dW, beta, ws, (size_t)ws_bytes, (int32_t*)info, st);
  Py_END_ALLOW_THREADS
  PyBuffer_Release(&off);
  return PyLong_FromLong(s);
}

/* sampled(X, dY, offsets, rows, A, lam, coeffs, ws, info, F2 or None) */
static PyObject* sampled(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  Operands o;
  Py_buffer off, rows;
  void *A, *c, *ws, *info, *F2 = NULL, *st;
  long long ws_bytes;
  int B;
  float lam;
  if (n != 10 || offsets(a[2], &off, &B)) return giving_up();
  if (int64_row(a[3], &rows)) {
    PyBuffer_Release(&off);
    return giving_up();
  }
  PyObject* result = NULL;
  if (!operands(a[0], a[1], 1, &o) && !vector(a[4], dt_f32, B, &A) && !float_arg(a[5], &lam) && !vector(a[6], dt_f32, B, &c) &&
      !address(a[7], &ws) && !call_int(a[7], s_numel, &ws_bytes) && !address(a[8], &info) &&
      (a[9] == Py_None || !vector(a[9], dt_f32, B, &F2)) && !stream(&st)) {
    isopo_status s;
    Py_BEGIN_ALLOW_THREADS
    s = lib.sampled(o.X, o.dY, o.dtype, o.T, (int)o.d_in, (int)o.d_out, (const int64_t*)off.buf, B, (const int64_t*)rows.buf,
                    (int)rows.shape[0], (const float*)A, lam, (float*)c, (float*)F2, ws, (size_t)ws_bytes, (int32_t*)info, st);
    Py_END_ALLOW_THREADS
    result = PyLong_FromLong(s);
  }
  PyBuffer_Release(&rows);
  PyBuffer_Release(&off);
  return result ? result : giving_up();
}

/* K, A, coeffs of a transform */
static int solve_args(PyObject* K, PyObject* A, PyObject* coeffs, PyObject* info, int* B, void** p) {
  long long nA;
  if (call_int(A, s_numel, &nA) || nA > INT32_MAX) return -1;
  *B = (int)nA;
  return !contiguous(K) || vector(K, dt_f32, nA * nA, &p[0]) || vector(A, dt_f32, -1, &p[1]) ||
                 vector(coeffs, dt_f32, nA, &p[2]) || address(info, &p[3])
             ? -1 : 0;
}

/* transform(K, A, variant, lam, coeffs, info) */
static PyObject* transform(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *p[4], *st;
  int B, variant;
  float lam;
  if (n != 6 || int_arg(a[2], &variant) || float_arg(a[3], &lam) || solve_args(a[0], a[1], a[4], a[5], &B, p) || stream(&st))
    return giving_up();
  isopo_status s;
  Py_BEGIN_ALLOW_THREADS
  s = lib.transform((const float*)p[0], (const float*)p[1], B, (isopo_variant)variant, lam, NULL, (float*)p[2], (int32_t*)p[3], st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(s);
}

/* transform_rel(K, A, variant, factor, state, coeffs, info) */
static PyObject* transform_rel(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *p[4], *state, *st;
  int B, variant;
  float factor;
  if (n != 7 || int_arg(a[2], &variant) || float_arg(a[3], &factor) || solve_args(a[0], a[1], a[5], a[6], &B, p) ||
      vector(a[4], dt_f32, 4, &state) || stream(&st))
    return giving_up();
  isopo_status s;
  Py_BEGIN_ALLOW_THREADS
  s = lib.transform_rel((const float*)p[0], (const float*)p[1], B, (isopo_variant)variant, factor, NULL, (const float*)state,
                        (float*)p[2], (int32_t*)p[3], st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(s);
}

/* reg_ema(K, decay, state) */
static PyObject* reg_ema(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  void *K, *state, *st;
  long long rows, cols;
  float decay;
  if (n != 3 || float_arg(a[1], &decay) || matrix_shape(a[0], &rows, &cols) || rows != cols || !contiguous(a[0]) ||
      vector(a[0], dt_f32, -1, &K) || !on_cuda(a[2]) || vector(a[2], dt_f32, 4, &state) || stream(&st))
    return giving_up();
  isopo_status s;
  Py_BEGIN_ALLOW_THREADS
  s = lib.reg_ema((const float*)K, (int)rows, decay, (float*)state, st);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(s);
}

/* bind(addresses of the library's functions in the order of `lib`, torch's dtypes, device and stream getters) */
static PyObject* bind(PyObject* self, PyObject* args) {
  unsigned long long f[6];
  PyObject *d[4], *g[2];
  if (!PyArg_ParseTuple(args, "(KKKKKK)(OOOO)(OO)", &f[0], &f[1], &f[2], &f[3], &f[4], &f[5], &d[0], &d[1], &d[2], &d[3],
                        &g[0], &g[1]))
    return NULL;
  memcpy(&lib.layer_gram, &f[0], sizeof(void*));
  memcpy(&lib.transform, &f[1], sizeof(void*));
  memcpy(&lib.transform_rel, &f[2], sizeof(void*));
  memcpy(&lib.reg_ema, &f[3], sizeof(void*));
  memcpy(&lib.weight_grad, &f[4], sizeof(void*));
  memcpy(&lib.sampled, &f[5], sizeof(void*));
  dt_f32 = Py_NewRef(d[0]);
  dt_bf16 = Py_NewRef(d[1]);
  dt_i32 = Py_NewRef(d[2]);
  dt_u8 = Py_NewRef(d[3]);
  get_device = Py_NewRef(g[0]);
  get_stream = Py_NewRef(g[1]);
  Py_RETURN_NONE;
}

static PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, NULL},
    {"layer_gram", (PyCFunction)(void (*)(void))layer_gram, METH_FASTCALL, NULL},
    {"transform", (PyCFunction)(void (*)(void))transform, METH_FASTCALL, NULL},
    {"transform_rel", (PyCFunction)(void (*)(void))transform_rel, METH_FASTCALL, NULL},
    {"reg_ema", (PyCFunction)(void (*)(void))reg_ema, METH_FASTCALL, NULL},
    {"sampled", (PyCFunction)(void (*)(void))sampled, METH_FASTCALL, NULL},
    {"weight_grad", (PyCFunction)(void (*)(void))weight_grad, METH_FASTCALL, NULL},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_calls", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__calls(void) {
  if (!(s_data_ptr = PyUnicode_InternFromString("data_ptr")) || !(s_dtype = PyUnicode_InternFromString("dtype")) ||
      !(s_is_cuda = PyUnicode_InternFromString("is_cuda")) || !(s_is_contiguous = PyUnicode_InternFromString("is_contiguous")) ||
      !(s_numel = PyUnicode_InternFromString("numel")) || !(s_shape = PyUnicode_InternFromString("shape")))
    return NULL;
  return PyModule_Create(&module);
}
