/* mikv_pycall.c — the Python binding's two decode-path calls in C: mikv_decode_step and mikv_decode_attention with
 * their tensors' pointers, checks and sizes gathered here instead of one ctypes argument at a time.
 *
 * A decode step takes nineteen tensors; fetching their pointers and converting the arguments in Python took most of
 * the 18 us that a step of a small cache spends on the host (its kernels run 10 us). Nothing is kept between calls but
 * the functions' addresses: every pointer is read, and every tensor checked, on every call. Compiled only where
 * Python's headers are installed; the ctypes path makes the same calls without it.
 */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>
#include <string.h>

#include "../../include/mikv.h"

typedef mikv_status (*step_fn)(const mikv_shape*, const mikv_cache*, int32_t, const void*, const void*, const void*,
                               int32_t, int32_t*, float, void*, int32_t, void*, size_t, void*);
typedef mikv_status (*attention_fn)(const mikv_shape*, const mikv_cache*, int32_t, const void*, float, void*, int32_t,
                                    float*, float*, void*, size_t, void*);

static step_fn g_step;
static attention_fn g_attention;
static PyObject* g_float32;  /* torch.float32 */
static PyObject *s_is_cuda, *s_is_contiguous, *s_data_ptr, *s_numel, *s_dtype, *s_shape, *s_packed;

enum { kArrays = 12 };
static const char* const kNames[kArrays] = {"k_hi",     "v_hi",     "hi_tok", "acc",      "k_codes",     "v_codes",
                                            "k_params", "v_params", "lo_tok", "balancer", "k_hi_params", "v_hi_params"};
static PyObject* s_names[kArrays];

/* The device address of tensor t (NULL for None); -1 with an exception for one that is not on a GPU or not contiguous. */
static int address(PyObject* t, void** out) {
  *out = NULL;
  if (t == Py_None) return 0;
  PyObject* v = PyObject_GetAttr(t, s_is_cuda);
  if (!v) return -1;
  int ok = PyObject_IsTrue(v);
  Py_DECREF(v);
  if (ok < 0) return -1;
  if (!ok) {
    PyErr_SetString(PyExc_ValueError, "libmikv takes device tensors");
    return -1;
  }
  v = PyObject_CallMethodNoArgs(t, s_is_contiguous);
  if (!v) return -1;
  ok = PyObject_IsTrue(v);
  Py_DECREF(v);
  if (ok < 0) return -1;
  if (!ok) {
    PyErr_SetString(PyExc_ValueError, "libmikv takes contiguous tensors");
    return -1;
  }
  v = PyObject_CallMethodNoArgs(t, s_data_ptr);
  if (!v) return -1;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return *out == NULL && PyErr_Occurred() ? -1 : 0;
}

static int shape_and_arrays(PyObject* cache, mikv_shape* shape, mikv_cache* arrays) {
  PyObject* s = PyObject_GetAttr(cache, s_shape);
  if (!s) return -1;
  PyObject* packed = PyObject_GetAttr(s, s_packed);
  Py_DECREF(s);
  if (!packed) return -1;
  if (!PyBytes_Check(packed) || PyBytes_GET_SIZE(packed) != (Py_ssize_t)sizeof *shape) {
    Py_DECREF(packed);
    PyErr_SetString(PyExc_TypeError, "packed shape");
    return -1;
  }
  memcpy(shape, PyBytes_AS_STRING(packed), sizeof *shape);
  Py_DECREF(packed);
  void* p[kArrays];
  for (int i = 0; i < kArrays; ++i) {
    PyObject* t = PyObject_GetAttr(cache, s_names[i]);
    if (!t) return -1;
    const int e = address(t, &p[i]);
    Py_DECREF(t);
    if (e) return -1;
  }
  _Static_assert(sizeof(mikv_cache) == kArrays * sizeof(void*), "twelve pointers");
  memcpy(arrays, p, sizeof p);
  return 0;
}

static int int32_of(PyObject* o, int32_t* out) {
  PyObject* i = PyNumber_Index(o);
  if (!i) return -1;
  const unsigned long v = PyLong_AsUnsignedLongMask(i);  /* the low bits, as a C int argument of ctypes */
  Py_DECREF(i);
  if (v == (unsigned long)-1 && PyErr_Occurred()) return -1;
  *out = (int32_t)(uint32_t)v;
  return 0;
}

static int out_and_workspace(PyObject* out, PyObject* ws, void** out_p, int32_t* out_dtype, void** ws_p, size_t* bytes) {
  PyObject* d = PyObject_GetAttr(out, s_dtype);
  if (!d) return -1;
  *out_dtype = d == g_float32 ? MIKV_OUT_F32 : MIKV_OUT_BF16;
  Py_DECREF(d);
  if (address(out, out_p) || address(ws, ws_p)) return -1;
  PyObject* n = PyObject_CallMethodNoArgs(ws, s_numel);
  if (!n) return -1;
  *bytes = PyLong_AsSize_t(n);
  Py_DECREF(n);
  return *bytes == (size_t)-1 && PyErr_Occurred() ? -1 : 0;
}

static int stream_of(PyObject* o, void** stream) {
  *stream = PyLong_AsVoidPtr(o);
  return *stream == NULL && PyErr_Occurred() ? -1 : 0;
}

/* decode_step(cache, n_lo, q, k_new, v_new, tok, slots, sm_scale, out, workspace, stream) -> status */
static PyObject* decode_step(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  mikv_shape shape;
  mikv_cache arrays;
  int32_t n_lo, tok, out_dtype;
  void *q, *k, *v, *slots, *out, *ws, *stream;
  size_t bytes;
  if (n != 11) {
    PyErr_SetString(PyExc_TypeError, "decode_step takes 11 arguments");
    return NULL;
  }
  if (shape_and_arrays(a[0], &shape, &arrays) || int32_of(a[1], &n_lo) || address(a[2], &q) || address(a[3], &k) ||
      address(a[4], &v) || int32_of(a[5], &tok) || address(a[6], &slots))
    return NULL;
  const double scale = PyFloat_AsDouble(a[7]);
  if (scale == -1.0 && PyErr_Occurred()) return NULL;
  if (out_and_workspace(a[8], a[9], &out, &out_dtype, &ws, &bytes) || stream_of(a[10], &stream)) return NULL;
  mikv_status rc;
  Py_BEGIN_ALLOW_THREADS
  rc = g_step(&shape, &arrays, n_lo, q, k, v, tok, (int32_t*)slots, (float)scale, out, out_dtype, ws, bytes, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)rc);
}

/* decode_attention(cache, n_lo, q, sm_scale, out, hi_logits, ml, workspace, stream) -> status */
static PyObject* decode_attention(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  mikv_shape shape;
  mikv_cache arrays;
  int32_t n_lo, out_dtype;
  void *q, *out, *logits, *ml, *ws, *stream;
  size_t bytes;
  if (n != 9) {
    PyErr_SetString(PyExc_TypeError, "decode_attention takes 9 arguments");
    return NULL;
  }
  if (shape_and_arrays(a[0], &shape, &arrays) || int32_of(a[1], &n_lo) || address(a[2], &q)) return NULL;
  const double scale = PyFloat_AsDouble(a[3]);
  if (scale == -1.0 && PyErr_Occurred()) return NULL;
  if (address(a[5], &logits) || address(a[6], &ml) || out_and_workspace(a[4], a[7], &out, &out_dtype, &ws, &bytes) ||
      stream_of(a[8], &stream))
    return NULL;
  mikv_status rc;
  Py_BEGIN_ALLOW_THREADS
  rc = g_attention(&shape, &arrays, n_lo, q, (float)scale, out, out_dtype, (float*)logits, (float*)ml, ws, bytes, stream);
  Py_END_ALLOW_THREADS
  return PyLong_FromLong((long)rc);
}

/* bind(step address, attention address, torch.float32) */
static PyObject* bind(PyObject* self, PyObject* args) {
  (void)self;
  PyObject *step, *attention, *f32;
  if (!PyArg_ParseTuple(args, "OOO", &step, &attention, &f32)) return NULL;
  void* ps = PyLong_AsVoidPtr(step);
  void* pa = PyLong_AsVoidPtr(attention);
  if (!ps || !pa) {
    if (!PyErr_Occurred()) PyErr_SetString(PyExc_ValueError, "null function");
    return NULL;
  }
  memcpy(&g_step, &ps, sizeof ps);
  memcpy(&g_attention, &pa, sizeof pa);
  Py_INCREF(f32);
  Py_XSETREF(g_float32, f32);
  Py_RETURN_NONE;
}

static PyMethodDef kMethods[] = {
    {"decode_step", (PyCFunction)(void (*)(void))decode_step, METH_FASTCALL, NULL},
    {"decode_attention", (PyCFunction)(void (*)(void))decode_attention, METH_FASTCALL, NULL},
    {"bind", bind, METH_VARARGS, NULL},
    {NULL, NULL, 0, NULL}};

static struct PyModuleDef kModule = {PyModuleDef_HEAD_INIT, "mikv_pycall", NULL, -1, kMethods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit_mikv_pycall(void) {
  static const struct {
    PyObject** to;
    const char* name;
  } names[] = {{&s_is_cuda, "is_cuda"}, {&s_is_contiguous, "is_contiguous"}, {&s_data_ptr, "data_ptr"},
               {&s_numel, "numel"},     {&s_dtype, "dtype"},                 {&s_shape, "shape"},
               {&s_packed, "packed"}};
  for (size_t i = 0; i < sizeof names / sizeof names[0]; ++i)
    if (!(*names[i].to = PyUnicode_InternFromString(names[i].name))) return NULL;
  for (int i = 0; i < kArrays; ++i)
    if (!(s_names[i] = PyUnicode_InternFromString(kNames[i]))) return NULL;
  return PyModule_Create(&kModule);
}
