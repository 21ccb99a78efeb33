/* The per-layer entry points of libdiffpro.so as CPython functions: marshalling only. A ctypes call with thirteen
 * arguments costs 1.5 us before the library sees it and the Python around it (pointers, sizes, the current
 * stream) another 1.5, next to 2.3 us for a launch: a one-launch call took 5.9 us of host time, 4.3 this way (the
 * adaLN layer for one token 6.0 -> 5.2 us a call, proj at 256 tokens 8.0 -> 6.7).
 * The functions' addresses, torch's stream lookup and the structures' types are handed in once by the binding (bind). */
#define PY_SSIZE_T_CLEAN
#include <Python.h>
#include <stdint.h>

#include "../../include/diffpro.h"

static int (*f_linear)(const dp_weight*, const void*, int64_t, const float*, int64_t, void*, int64_t, void*, size_t,
                       const dp_debug*, int32_t*, uint32_t, dp_stream);
static int (*f_residual)(const dp_weight*, const void*, int64_t, int64_t, const dp_residual*, void*, int64_t, void*,
                         size_t, int32_t*, uint32_t, dp_stream);
static int (*f_daq)(const void*, int64_t, int64_t, int64_t, int8_t*, int64_t, float*, int32_t*, dp_stream);
static int (*f_ln)(const void*, int64_t, int64_t, int64_t, const void*, const void*, int64_t, float, int8_t*, int64_t,
                   float*, dp_stream);
static PyObject *g_get_device, *g_get_stream; /* torch.cuda.current_device, torch._C._cuda_getCurrentRawStream */
static PyObject *g_weight, *g_debug, *g_arg_error; /* the ctypes structures dp_weight and dp_debug, ctypes.ArgumentError */
static PyObject *s_data_ptr, *s_nbytes, *s_cuda_stream;

/* The converters leave a Python error behind; callers look once, before the call, with PyErr_Occurred. */
static void* as_ptr(PyObject* v) {
  void* p = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return p;
}
static void* tensor_ptr(PyObject* t) { /* a tensor or None */
  if (t == Py_None || PyErr_Occurred()) return NULL;
  PyObject* v = PyObject_CallMethodNoArgs(t, s_data_ptr);
  return v ? as_ptr(v) : NULL;
}
static size_t tensor_bytes(PyObject* t) {
  if (t == Py_None || PyErr_Occurred()) return 0;
  PyObject* v = PyObject_GetAttr(t, s_nbytes);
  if (!v) return 0;
  const size_t n = PyLong_AsSize_t(v);
  Py_DECREF(v);
  return n;
}
static dp_stream stream_of(PyObject* s) { /* a torch stream, or None: the current one */
  if (PyErr_Occurred()) return NULL;
  PyObject* v;
  if (s == Py_None) {
    PyObject* dev = PyObject_CallNoArgs(g_get_device);
    if (!dev) return NULL;
    v = PyObject_CallOneArg(g_get_stream, dev);
    Py_DECREF(dev);
  } else {
    v = PyObject_GetAttr(s, s_cuda_stream);
  }
  return v ? (dp_stream)as_ptr(v) : NULL;
}
static int64_t as_i64(PyObject* o) { return PyErr_Occurred() ? 0 : PyLong_AsLongLong(o); }
static void* as_addr(PyObject* o) { return PyErr_Occurred() ? NULL : PyLong_AsVoidPtr(o); }
/* The memory of a ctypes structure, which has to be of that type: another one's would be read past its end. */
static void* as_struct(PyObject* o, PyObject* type) {
  Py_buffer b;
  if (PyErr_Occurred()) return NULL;
  if (!PyObject_TypeCheck(o, (PyTypeObject*)type)) {
    PyErr_Format(g_arg_error, "expected %s instance instead of %s", ((PyTypeObject*)type)->tp_name, Py_TYPE(o)->tp_name);
    return NULL;
  }
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE)) return NULL;
  void* p = b.buf;
  PyBuffer_Release(&b); /* (the caller's reference keeps it) */
  return p;
}
static uint32_t as_flags(PyObject* o) { return PyErr_Occurred() ? 0 : (uint32_t)PyLong_AsUnsignedLongMask(o); }

static int args_ok(Py_ssize_t n, Py_ssize_t want) {
  if (n == want && g_get_stream) return 1;
  PyErr_Format(PyExc_TypeError, "%zd arguments wanted, %zd given (or bind not called)", want, n);
  return 0;
}

/* (weight, x, ldx, s_a_in, M, y, ldy, workspace, debug or None, device_status, flags, stream) */
static PyObject* wq_linear(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  if (!args_ok(n, 12)) return NULL;
  const dp_weight* w = as_struct(a[0], g_weight);
  const void* x = tensor_ptr(a[1]);
  const int64_t ldx = as_i64(a[2]);
  const float* sa = tensor_ptr(a[3]);
  const int64_t M = as_i64(a[4]);
  void* y = tensor_ptr(a[5]);
  const int64_t ldy = as_i64(a[6]);
  void* ws = tensor_ptr(a[7]);
  const size_t wsb = tensor_bytes(a[7]);
  const dp_debug* dbg = a[8] == Py_None ? NULL : as_struct(a[8], g_debug);
  int32_t* status = tensor_ptr(a[9]);
  const uint32_t flags = as_flags(a[10]);
  const dp_stream s = stream_of(a[11]);
  if (PyErr_Occurred()) return NULL;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_linear(w, x, ldx, sa, M, y, ldy, ws, wsb, dbg, status, flags, s);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

/* (weight, x, ldx, M, residual, ldr, gate, rows_per_gate, y, ldy, workspace, ws_bytes, device_status, flags,
 * stream) */
static PyObject* wq_linear_residual(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  if (!args_ok(n, 15)) return NULL;
  const dp_weight* w = as_struct(a[0], g_weight);
  const void* x = tensor_ptr(a[1]);
  const int64_t ldx = as_i64(a[2]), M = as_i64(a[3]);
  dp_residual r;
  r.residual = tensor_ptr(a[4]);
  r.ldr = as_i64(a[5]);
  r.gate = tensor_ptr(a[6]);
  r.rows_per_gate = as_i64(a[7]);
  void* y = tensor_ptr(a[8]);
  const int64_t ldy = as_i64(a[9]);
  void* ws = tensor_ptr(a[10]);
  const int64_t wsb = as_i64(a[11]);
  int32_t* status = tensor_ptr(a[12]);
  const uint32_t flags = as_flags(a[13]);
  const dp_stream s = stream_of(a[14]);
  if (PyErr_Occurred()) return NULL;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_residual(w, x, ldx, M, &r, y, ldy, ws, (size_t)wsb, status, flags, s);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

/* (x, M, K, ldx, q, ldq, s_a, rowsum, stream) */
static PyObject* daq_quantize(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  if (!args_ok(n, 9)) return NULL;
  const void* x = tensor_ptr(a[0]);
  const int64_t M = as_i64(a[1]), K = as_i64(a[2]), ldx = as_i64(a[3]);
  int8_t* q = tensor_ptr(a[4]);
  const int64_t ldq = as_i64(a[5]);
  float* sa = tensor_ptr(a[6]);
  int32_t* rowsum = tensor_ptr(a[7]);
  const dp_stream s = stream_of(a[8]);
  if (PyErr_Occurred()) return NULL;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_daq(x, M, K, ldx, q, ldq, sa, rowsum, s);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

/* (x, M, K, ldx, shift, scale, rows_per_sample, eps, q, ldq, s_a, stream) */
static PyObject* ln_modulate_daq(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  if (!args_ok(n, 12)) return NULL;
  const void* x = tensor_ptr(a[0]);
  const int64_t M = as_i64(a[1]), K = as_i64(a[2]), ldx = as_i64(a[3]);
  const void *shift = tensor_ptr(a[4]), *scale = tensor_ptr(a[5]);
  const int64_t rps = as_i64(a[6]);
  const double eps = PyErr_Occurred() ? 0.0 : PyFloat_AsDouble(a[7]);
  int8_t* q = tensor_ptr(a[8]);
  const int64_t ldq = as_i64(a[9]);
  float* sa = tensor_ptr(a[10]);
  const dp_stream s = stream_of(a[11]);
  if (PyErr_Occurred()) return NULL;
  int st;
  Py_BEGIN_ALLOW_THREADS;
  st = f_ln(x, M, K, ldx, shift, scale, rps, (float)eps, q, ldq, sa, s);
  Py_END_ALLOW_THREADS;
  return PyLong_FromLong(st);
}

/* (addresses of dp_wq_linear, dp_wq_linear_residual, dp_daq_quantize, dp_ln_modulate_daq, device getter, stream getter,
 * dp_weight, dp_debug, ctypes.ArgumentError) */
static PyObject* bind(PyObject* self, PyObject* const* a, Py_ssize_t n) {
  (void)self;
  if (n != 9 || !PyType_Check(a[6]) || !PyType_Check(a[7])) {
    PyErr_SetString(PyExc_TypeError, "bind takes four addresses, two callables and three types");
    return NULL;
  }
  void* p[4];
  for (int i = 0; i < 4; ++i) p[i] = as_addr(a[i]);
  if (PyErr_Occurred()) return NULL;
  *(void**)&f_linear = p[0];
  *(void**)&f_residual = p[1];
  *(void**)&f_daq = p[2];
  *(void**)&f_ln = p[3];
  PyObject** keep[5] = {&g_get_device, &g_get_stream, &g_weight, &g_debug, &g_arg_error};
  for (int i = 0; i < 5; ++i) {
    Py_INCREF(a[4 + i]);
    Py_XSETREF(*keep[i], a[4 + i]);
  }
  Py_RETURN_NONE;
}

#define FAST(f) (PyCFunction)(void (*)(void))f, METH_FASTCALL, NULL
static PyMethodDef methods[] = {{"bind", FAST(bind)},
                                {"wq_linear", FAST(wq_linear)},
                                {"wq_linear_residual", FAST(wq_linear_residual)},
                                {"daq_quantize", FAST(daq_quantize)},
                                {"ln_modulate_daq", FAST(ln_modulate_daq)},
                                {NULL, NULL, 0, NULL}};
static struct PyModuleDef module = {PyModuleDef_HEAD_INIT, "_call", NULL, -1, methods, NULL, NULL, NULL, NULL};

PyMODINIT_FUNC PyInit__call(void) {
  s_data_ptr = PyUnicode_InternFromString("data_ptr");
  s_nbytes = PyUnicode_InternFromString("nbytes");
  s_cuda_stream = PyUnicode_InternFromString("cuda_stream");
  if (!s_data_ptr || !s_nbytes || !s_cuda_stream) return NULL;
  return PyModule_Create(&module);
}
