/* Python entry points of the calls that a program makes per layer: the same names and arguments as their wrappers in binding.py,
 * marshalled here instead of through ctypes.  A small layer's kernels take 4 to 8 us; the wrappers took 4 us per call to look at
 * their arguments one by one in Python and to convert them (per-token quantizer and layer of 64 x 1152 x 1152: 13.8 us per pass, now 7.8;
 * attention of 6 heads with 64 tokens 6.9, now 4.1).
 *
 * Only the ordinary call is served: positional arguments that are tensors (anything with data_ptr()), Python ints and floats, None and
 * the binding's own structures.  Every other call (keywords, numpy arrays, a wrong number or type of arguments) goes to the wrapper,
 * and a status other than QDIT_OK to its check(), so that both accept, refuse and raise the same. */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "qdit.h"

enum { QUANTIZE_ACT, W8A8_LINEAR, W4A8_LINEAR, ATTENTION, ADALN_MODULATE, CALLS };

static void* g_call[CALLS];          /* the library's functions */
static PyObject* g_wrapper[CALLS];   /* the wrappers of the same names */
static PyObject *g_check, *g_data_ptr, *g_zero;
static PyTypeObject *g_qparams, *g_epilogue;

/* Converters: 1, or 0 (without an exception) if the argument is not of the ordinary kind. */
static int to_ptr(PyObject* o, void** out) {
  if (o == Py_None) {
    *out = NULL;
    return 1;
  }
  PyObject* address = NULL;
  if (!PyLong_CheckExact(o)) {
    address = o = PyObject_CallMethodNoArgs(o, g_data_ptr);
    if (!o || !PyLong_CheckExact(o)) {
      Py_XDECREF(address);
      PyErr_Clear();
      return 0;
    }
  }
  *out = PyLong_AsVoidPtr(o);
  const int ok = !(*out == NULL && PyErr_Occurred());
  PyErr_Clear();
  Py_XDECREF(address);
  return ok;
}
static int to_i64(PyObject* o, int64_t* out) {
  if (!PyLong_CheckExact(o)) return 0;
  int overflow;
  *out = PyLong_AsLongLongAndOverflow(o, &overflow);
  return !overflow;
}
static int to_i32(PyObject* o, int* out) {
  int64_t v;
  if (!to_i64(o, &v) || v < INT32_MIN || v > INT32_MAX) return 0;
  *out = (int)v;
  return 1;
}
static int to_u32(PyObject* o, uint32_t* out) {
  int64_t v;
  if (!to_i64(o, &v) || v < 0 || v > UINT32_MAX) return 0;
  *out = (uint32_t)v;
  return 1;
}
static int to_f32(PyObject* o, float* out) {
  if (!PyFloat_CheckExact(o)) return 0;
  *out = (float)PyFloat_AS_DOUBLE(o);
  return 1;
}
/* A copy of one of the binding's structures, which another thread may change while the call runs; *given = 0 for None. */
static int to_struct(PyObject* o, PyTypeObject* type, void* copy, Py_ssize_t size, int* given) {
  *given = o != Py_None;
  if (!*given) return 1;
  Py_buffer view;
  if (Py_TYPE(o) != type || PyObject_GetBuffer(o, &view, PyBUF_SIMPLE) != 0) {
    PyErr_Clear();
    return 0;
  }
  const int ok = view.len == size;
  if (ok) memcpy(copy, view.buf, (size_t)size);
  PyBuffer_Release(&view);
  return ok;
}

static PyObject* done(PyObject* ctx, int32_t status) {
  if (status == QDIT_OK) return Py_NewRef(g_zero);
  return PyObject_CallFunction(g_check, "Oi", ctx, (int)status);
}
#define WRAPPER(i) return PyObject_Vectorcall(g_wrapper[i], a, (size_t)n, names)

static PyObject* quantize_act(PyObject* self, PyObject* const* a, Py_ssize_t n, PyObject* names) {
  void *ctx, *x, *scale, *q;
  int dtype, mode, given;
  int64_t M, K, ldx, ldq;
  qdit_qparams qp;
  if (n != 11 || names || !to_ptr(a[0], &ctx) || !to_ptr(a[1], &x) || !to_i32(a[2], &dtype) || !to_i64(a[3], &M) || !to_i64(a[4], &K) ||
      !to_i64(a[5], &ldx) || !to_i32(a[6], &mode) || !to_struct(a[7], g_qparams, &qp, sizeof(qp), &given) || !to_ptr(a[8], &scale) ||
      !to_ptr(a[9], &q) || !to_i64(a[10], &ldq))
    WRAPPER(QUANTIZE_ACT);
  int32_t st;
  Py_BEGIN_ALLOW_THREADS
  st = ((int32_t (*)(qdit_ctx*, const void*, int, int64_t, int64_t, int64_t, int, const qdit_qparams*, float*, void*, int64_t))g_call[QUANTIZE_ACT])(
      ctx, x, dtype, M, K, ldx, mode, given ? &qp : NULL, scale, q, ldq);
  Py_END_ALLOW_THREADS
  return done(a[0], st);
}

static PyObject* linear(int which, PyObject* const* a, Py_ssize_t n, PyObject* names) {
  void *ctx, *A, *W, *a_scale, *out, *scratch = NULL;
  int64_t M, N, K, ldo;
  uint32_t flags;
  int given_qp, given_epi;
  qdit_qparams qp;
  qdit_epilogue epi;
  if (!(n == 12 || (n == 13 && which == W4A8_LINEAR)) || names || !to_ptr(a[0], &ctx) || !to_ptr(a[1], &A) || !to_ptr(a[2], &W) ||
      !to_i64(a[3], &M) || !to_i64(a[4], &N) || !to_i64(a[5], &K) || !to_struct(a[6], g_qparams, &qp, sizeof(qp), &given_qp) || !given_qp ||
      !to_ptr(a[7], &a_scale) || !to_u32(a[8], &flags) || !to_struct(a[9], g_epilogue, &epi, sizeof(epi), &given_epi) ||
      !to_ptr(a[10], &out) || !to_i64(a[11], &ldo) || (n == 13 && !to_ptr(a[12], &scratch)))
    WRAPPER(which);
  int32_t st;
  Py_BEGIN_ALLOW_THREADS
  if (which == W4A8_LINEAR)
    st = ((int32_t (*)(qdit_ctx*, const void*, const void*, int64_t, int64_t, int64_t, qdit_qparams, const float*, uint32_t, const qdit_epilogue*, void*,
                       int64_t, void*))g_call[W4A8_LINEAR])(ctx, A, W, M, N, K, qp, a_scale, flags, given_epi ? &epi : NULL, out, ldo, scratch);
  else
    st = ((int32_t (*)(qdit_ctx*, const void*, const void*, int64_t, int64_t, int64_t, qdit_qparams, const float*, uint32_t, const qdit_epilogue*, void*,
                       int64_t))g_call[W8A8_LINEAR])(ctx, A, W, M, N, K, qp, a_scale, flags, given_epi ? &epi : NULL, out, ldo);
  Py_END_ALLOW_THREADS
  return done(a[0], st);
}
static PyObject* w8a8_linear(PyObject* self, PyObject* const* a, Py_ssize_t n, PyObject* names) { return linear(W8A8_LINEAR, a, n, names); }
static PyObject* w4a8_linear(PyObject* self, PyObject* const* a, Py_ssize_t n, PyObject* names) { return linear(W4A8_LINEAR, a, n, names); }

static PyObject* attention(PyObject* self, PyObject* const* a, Py_ssize_t n, PyObject* names) {
  void *ctx, *q, *k, *v, *out, *scale = NULL;
  int64_t ld;
  int B, H, T, dh, dtype, given = 0;
  float softmax_scale;
  qdit_qparams qp;
  if (n < 12 || n > 14 || names || !to_ptr(a[0], &ctx) || !to_ptr(a[1], &q) || !to_ptr(a[2], &k) || !to_ptr(a[3], &v) || !to_i64(a[4], &ld) ||
      !to_i32(a[5], &B) || !to_i32(a[6], &H) || !to_i32(a[7], &T) || !to_i32(a[8], &dh) || !to_f32(a[9], &softmax_scale) ||
      !to_ptr(a[10], &out) || !to_i32(a[11], &dtype) || (n > 12 && !to_struct(a[12], g_qparams, &qp, sizeof(qp), &given)) ||
      (n > 13 && !to_ptr(a[13], &scale)))
    WRAPPER(ATTENTION);
  int32_t st;
  Py_BEGIN_ALLOW_THREADS
  st = ((int32_t (*)(qdit_ctx*, const void*, const void*, const void*, int64_t, int, int, int, int, float, void*, int, const qdit_qparams*,
                     const float*))g_call[ATTENTION])(ctx, q, k, v, ld, B, H, T, dh, softmax_scale, out, dtype, given ? &qp : NULL, scale);
  Py_END_ALLOW_THREADS
  return done(a[0], st);
}

static PyObject* adaln_modulate(PyObject* self, PyObject* const* a, Py_ssize_t n, PyObject* names) {
  void *ctx, *x, *shift, *scale, *out, *out_scale = NULL;
  int64_t M, D, T, ld;
  int dtype, given = 0;
  float eps;
  qdit_qparams qp;
  if (n < 11 || n > 13 || names || !to_ptr(a[0], &ctx) || !to_ptr(a[1], &x) || !to_i64(a[2], &M) || !to_i64(a[3], &D) || !to_i64(a[4], &T) ||
      !to_f32(a[5], &eps) || !to_ptr(a[6], &shift) || !to_ptr(a[7], &scale) || !to_i64(a[8], &ld) || !to_ptr(a[9], &out) ||
      !to_i32(a[10], &dtype) || (n > 11 && !to_struct(a[11], g_qparams, &qp, sizeof(qp), &given)) || (n > 12 && !to_ptr(a[12], &out_scale)))
    WRAPPER(ADALN_MODULATE);
  int32_t st;
  Py_BEGIN_ALLOW_THREADS
  st = ((int32_t (*)(qdit_ctx*, const void*, int64_t, int64_t, int64_t, float, const float*, const float*, int64_t, void*, int, const qdit_qparams*,
                     const float*))g_call[ADALN_MODULATE])(ctx, x, M, D, T, eps, shift, scale, ld, out, dtype, given ? &qp : NULL, out_scale);
  Py_END_ALLOW_THREADS
  return done(a[0], st);
}

/* bind(addresses of the library's functions, wrappers, check, qparams type, epilogue type); the first two in the order of the enum */
static PyObject* bind(PyObject* self, PyObject* args) {
  PyObject *addresses, *wrappers, *check, *qparams, *epilogue;
  if (!PyArg_ParseTuple(args, "O!O!OO!O!", &PyTuple_Type, &addresses, &PyTuple_Type, &wrappers, &check, &PyType_Type, &qparams, &PyType_Type, &epilogue))
    return NULL;
  if (PyTuple_GET_SIZE(addresses) != CALLS || PyTuple_GET_SIZE(wrappers) != CALLS) {
    PyErr_SetString(PyExc_ValueError, "one address and one wrapper per call");
    return NULL;
  }
  for (int i = 0; i < CALLS; ++i) {
    g_call[i] = PyLong_AsVoidPtr(PyTuple_GET_ITEM(addresses, i));
    if (PyErr_Occurred()) return NULL;
    Py_XSETREF(g_wrapper[i], Py_NewRef(PyTuple_GET_ITEM(wrappers, i)));
  }
  Py_XSETREF(g_check, Py_NewRef(check));
  Py_XSETREF(g_qparams, (PyTypeObject*)Py_NewRef(qparams));
  Py_XSETREF(g_epilogue, (PyTypeObject*)Py_NewRef(epilogue));
  Py_RETURN_NONE;
}

#define FAST(name) (PyCFunction)(void (*)(void))name, METH_FASTCALL | METH_KEYWORDS
#define SIGNATURE_ENDS "\n--\n\n"   /* what makes the line a signature that inspect finds */
static PyMethodDef methods[] = {
    {"bind", bind, METH_VARARGS, "Sets the functions that the calls below reach."},
    {"qdit_quantize_act", FAST(quantize_act), "qdit_quantize_act(ctx, x, x_dtype, M, K, ldx, mode, qp, dyn_scale, q, ldq)" SIGNATURE_ENDS},
    {"qdit_w8a8_linear", FAST(w8a8_linear), "qdit_w8a8_linear(ctx, A, W, M, N, K, a_qp, a_scale_dev, flags, epi, out, ldo)" SIGNATURE_ENDS},
    {"qdit_w4a8_linear", FAST(w4a8_linear), "qdit_w4a8_linear(ctx, A, W_packed, M, N, K, a_qp, a_scale_dev, flags, epi, out, ldo, w8_scratch=None)" SIGNATURE_ENDS},
    {"qdit_attention", FAST(attention), "qdit_attention(ctx, q, k, v, ld, B, H, T, dh, softmax_scale, out, out_dtype, out_qp=None, out_scale_dev=None)" SIGNATURE_ENDS},
    {"qdit_adaln_modulate", FAST(adaln_modulate), "qdit_adaln_modulate(ctx, x, M, D, T, eps, shift, scale, ld_mod, out, out_dtype, out_qp=None, out_scale_dev=None)" SIGNATURE_ENDS},
    {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_marshal", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__marshal(void) {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  g_zero = PyLong_FromLong(0);
  if (!g_data_ptr || !g_zero) return NULL;
  return PyModule_Create(&module);
}
