// Native half of binding.py: argument marshalling between Python objects and the C ABI (adaption.h), and
// nothing else.  A layer call through ctypes cost 8 to 12 us of interpreter time in front of a launch, more
// than the small layers take on the GPU; here it costs about 1 us.
//
// The library itself is opened by path (bind), so that this module holds no link dependency on it.
// Tensors are read through their own attributes at every call (data_ptr() of the planes, formats,
// pitch): nothing about an argument is kept from one call to the next.  The interpreter lock is released
// around every call into the library.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <dlfcn.h>

#include <cstring>

#include "adaption.h"

namespace {

// the library's entry points
#define ADAPTION_FUNCTIONS(X)                                                                                        \
  X(adaption_measure_range) X(adaption_quantize) X(adaption_quantize_batch) X(adaption_quantize_batch_stochastic)    \
  X(adaption_quantize_stochastic) X(adaption_lp_act) X(adaption_lp_act_stochastic) X(adaption_bit_histogram)         \
  X(adaption_width_histogram) X(adaption_lp_conv_workspace_bytes) X(adaption_lp_conv_fwd)                            \
  X(adaption_lp_conv_fwd_stochastic) X(adaption_lp_conv_pool_workspace_bytes) X(adaption_lp_conv_pool_fwd)           \
  X(adaption_lp_ip_workspace_bytes) X(adaption_lp_ip_fwd) X(adaption_lp_ip_fwd_stochastic)                           \
  X(adaption_lp_ip_fwd_static_ws) X(adaption_maxpool2x2)
#define DECLARE(f) decltype(&::f) p_##f = nullptr;
ADAPTION_FUNCTIONS(DECLARE)
#undef DECLARE

PyObject* g_error = nullptr;        // AdaptionError
PyObject* g_device = nullptr;       // () -> current device ordinal
PyObject* g_stream = nullptr;       // (device) -> raw handle of the current stream

PyObject *s_lo, *s_hi, *s_q16, *s_n_bits, *s_frac_bits, *s_c_stride, *s_outer, *s_inner, *s_data_ptr, *s_numel, *s_itemsize;

bool attr_i64(PyObject* o, PyObject* name, long long* out) {
  PyObject* v = PyObject_GetAttr(o, name);
  if (v == nullptr) return false;
  *out = PyLong_AsLongLong(v);
  Py_DECREF(v);
  return !(*out == -1 && PyErr_Occurred());
}
// tensor (or None) -> device pointer
bool tensor_ptr(PyObject* t, void** out) {
  *out = nullptr;
  if (t == Py_None) return true;
  PyObject* v = PyObject_CallMethodNoArgs(t, s_data_ptr);
  if (v == nullptr) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return !(*out == nullptr && PyErr_Occurred());
}
bool attr_ptr(PyObject* o, PyObject* name, void** out) {
  PyObject* t = PyObject_GetAttr(o, name);
  if (t == nullptr) return false;
  const bool ok = tensor_ptr(t, out);
  Py_DECREF(t);
  return ok;
}
// QTensor -> descriptor
bool qtensor(PyObject* o, adaption_qtensor* q) {
  long long n, f, cs;
  void* q16;
  if (!attr_ptr(o, s_hi, &q->hi) || !attr_ptr(o, s_lo, &q->lo) || !attr_ptr(o, s_q16, &q16) || !attr_i64(o, s_n_bits, &n) ||
      !attr_i64(o, s_frac_bits, &f) || !attr_i64(o, s_c_stride, &cs))
    return false;
  q->q16 = static_cast<int16_t*>(q16);
  q->fmt.n_bits = (int32_t)n;
  q->fmt.frac_bits = (int32_t)f;
  q->c_stride = cs;
  return true;
}
bool i64(PyObject* o, long long* out) {
  *out = PyLong_AsLongLong(o);
  return !(*out == -1 && PyErr_Occurred());
}
bool i32(PyObject* o, int32_t* out) {
  long long v;
  if (!i64(o, &v)) return false;
  *out = (int32_t)v;
  return true;
}
bool truth(PyObject* o, int32_t* out) {
  const int t = PyObject_IsTrue(o);
  *out = t;
  return t >= 0;
}
bool u64(PyObject* o, uint64_t* out) {         // modulo 2^64
  PyObject* i = PyNumber_Index(o);
  if (i == nullptr) return false;
  *out = PyLong_AsUnsignedLongLongMask(i);
  Py_DECREF(i);
  return !PyErr_Occurred();
}
bool current_stream(void** out) {
  PyObject* d = PyObject_CallNoArgs(g_device);
  if (d == nullptr) return false;
  PyObject* s = PyObject_CallOneArg(g_stream, d);
  Py_DECREF(d);
  if (s == nullptr) return false;
  *out = PyLong_AsVoidPtr(s);
  Py_DECREF(s);
  return !(*out == nullptr && PyErr_Occurred());
}
bool numel(PyObject* t, long long* out) {
  PyObject* n = PyObject_CallMethodNoArgs(t, s_numel);
  if (n == nullptr) return false;
  *out = PyLong_AsLongLong(n);
  Py_DECREF(n);
  return !(*out == -1 && PyErr_Occurred());
}
// bytes of a tensor (workspace), 0 for None
bool workspace(PyObject* t, void** p, size_t* bytes) {
  *bytes = 0;
  if (!tensor_ptr(t, p)) return false;
  if (t == Py_None) return true;
  long long n, item;
  if (!numel(t, &n) || !attr_i64(t, s_itemsize, &item)) return false;
  *bytes = (size_t)(n * item);
  return true;
}
// read-only view of a ctypes structure
struct Buffer {
  Py_buffer b;
  bool held = false;
  ~Buffer() {
    if (held) PyBuffer_Release(&b);
  }
  bool get(PyObject* o, size_t need, const char* what, int flags = PyBUF_SIMPLE) {
    if (PyObject_GetBuffer(o, &b, flags) != 0) return false;
    held = true;
    if ((size_t)b.len < need) {
      PyErr_Format(PyExc_TypeError, "%s: a structure of %zu bytes is expected", what, need);
      return false;
    }
    return true;
  }
};

PyObject* answer(int rc, const char* where) {
  if (rc == ADAPTION_OK) Py_RETURN_NONE;
  PyObject* e = PyObject_CallFunction(g_error, "is", rc, where);
  if (e != nullptr) {
    PyErr_SetObject(g_error, e);
    Py_DECREF(e);
  }
  return nullptr;
}

#define ARGS(n)                                                                        \
  if (nargs != (n)) {                                                                  \
    PyErr_Format(PyExc_TypeError, "%d arguments expected, got %zd", (n), nargs);       \
    return nullptr;                                                                    \
  }
#define CALL(expr)            \
  int rc;                     \
  Py_BEGIN_ALLOW_THREADS rc = (expr); \
  Py_END_ALLOW_THREADS

// x, n_bits, d_max_abs, d_fmt_out
PyObject* measure_range(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(4)
  void *x, *mx, *fmt, *st;
  long long count;
  int32_t n;
  if (!tensor_ptr(a[0], &x) || !numel(a[0], &count) || !i32(a[1], &n) || !tensor_ptr(a[2], &mx) || !tensor_ptr(a[3], &fmt) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_measure_range((const float*)x, (size_t)count, n, (float*)mx, (adaption_qfmt*)fmt, st))
  return answer(rc, "adaption_measure_range");
}

// x, outer, inner, out, d_fmt, rounding, d_stats
PyObject* quantize(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(7)
  void *x, *fmt, *stats, *st;
  long long outer, inner;
  int32_t rounding;
  adaption_qtensor q;
  if (!tensor_ptr(a[0], &x) || !i64(a[1], &outer) || !i64(a[2], &inner) || !qtensor(a[3], &q) || !tensor_ptr(a[4], &fmt) ||
      !i32(a[5], &rounding) || !tensor_ptr(a[6], &stats) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_quantize((const float*)x, (size_t)outer, (size_t)inner, q, (const adaption_qfmt*)fmt, rounding,
                           (adaption_stats*)stats, st))
  return answer(rc, "adaption_quantize");
}

// items (ctypes array, filled here), entries: (x, outer, inner, out, d_fmt or None) each
PyObject* fill_items(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(2)
  PyObject* seq = PySequence_Fast(a[1], "a sequence of entries is expected");
  if (seq == nullptr) return nullptr;
  const Py_ssize_t n = PySequence_Fast_GET_SIZE(seq);
  Buffer b;
  bool ok = b.get(a[0], (size_t)n * sizeof(adaption_quantize_item), "items", PyBUF_WRITABLE);
  for (Py_ssize_t k = 0; ok && k < n; ++k) {
    adaption_quantize_item& it = static_cast<adaption_quantize_item*>(b.b.buf)[k];
    PyObject* e = PySequence_Fast(PySequence_Fast_GET_ITEM(seq, k), "an entry is a sequence");
    if (e == nullptr) { ok = false; break; }
    if (PySequence_Fast_GET_SIZE(e) != 5) {
      PyErr_SetString(PyExc_ValueError, "an entry is (x, outer, inner, out, d_fmt)");
      ok = false;
    } else {
      PyObject** v = PySequence_Fast_ITEMS(e);
      void *x, *fmt;
      long long outer, inner;
      ok = tensor_ptr(v[0], &x) && i64(v[1], &outer) && i64(v[2], &inner) && qtensor(v[3], &it.q) && tensor_ptr(v[4], &fmt);
      if (ok) {
        it.d_x = (const float*)x;
        it.outer = outer;
        it.inner = inner;
        it.d_fmt = (const adaption_qfmt*)fmt;
      }
    }
    Py_DECREF(e);
  }
  Py_DECREF(seq);
  if (!ok) return nullptr;
  Py_RETURN_NONE;
}

// items (None: a null pointer, which the library takes with n = 0 and refuses otherwise), n
PyObject* quantize_batch(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(2)
  int32_t n;
  void* st;
  Buffer b;
  if (!i32(a[1], &n) ||
      (a[0] != Py_None && !b.get(a[0], n > 0 ? (size_t)n * sizeof(adaption_quantize_item) : 0, "items")) ||
      !current_stream(&st))
    return nullptr;
  CALL(p_adaption_quantize_batch(b.held ? (const adaption_quantize_item*)b.b.buf : nullptr, n, st))
  return answer(rc, "adaption_quantize_batch");
}

// items, seeds (ctypes array of uint64), n
PyObject* quantize_batch_stochastic(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(3)
  int32_t n;
  void* st;
  Buffer b, s;
  if (!i32(a[2], &n) || !b.get(a[0], (size_t)n * sizeof(adaption_quantize_item), "items") ||
      !s.get(a[1], (size_t)n * sizeof(uint64_t), "seeds") || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_quantize_batch_stochastic((const adaption_quantize_item*)b.b.buf, (const uint64_t*)s.b.buf, n, st))
  return answer(rc, "adaption_quantize_batch_stochastic");
}

// x, outer, inner, out, seed, relu, d_fmt, d_stats
PyObject* quantize_stochastic(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(8)
  void *x, *fmt, *stats, *st;
  long long outer, inner;
  int32_t relu;
  uint64_t seed;
  adaption_qtensor q;
  if (!tensor_ptr(a[0], &x) || !i64(a[1], &outer) || !i64(a[2], &inner) || !qtensor(a[3], &q) || !u64(a[4], &seed) ||
      !truth(a[5], &relu) || !tensor_ptr(a[6], &fmt) || !tensor_ptr(a[7], &stats) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_quantize_stochastic((const float*)x, (size_t)outer, (size_t)inner, q, (const adaption_qfmt*)fmt, relu, seed,
                                      (adaption_stats*)stats, st))
  return answer(rc, "adaption_quantize_stochastic");
}

// x_f32, x_q, outer, inner, relu, out, d_fmt, rounding, d_stats
PyObject* lp_act(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(9)
  void *x, *fmt, *stats, *st;
  long long outer, inner;
  int32_t relu, rounding;
  adaption_qtensor xq, q;
  if (!tensor_ptr(a[0], &x) || (a[1] != Py_None && !qtensor(a[1], &xq)) || !i64(a[2], &outer) || !i64(a[3], &inner) ||
      !truth(a[4], &relu) || !qtensor(a[5], &q) || !tensor_ptr(a[6], &fmt) || !i32(a[7], &rounding) ||
      !tensor_ptr(a[8], &stats) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_lp_act((const float*)x, a[1] == Py_None ? nullptr : &xq, (size_t)outer, (size_t)inner, relu, q,
                         (const adaption_qfmt*)fmt, rounding, (adaption_stats*)stats, st))
  return answer(rc, "adaption_lp_act");
}

// x_f32, x_q, outer, inner, relu, out, seed, d_fmt, d_stats
PyObject* lp_act_stochastic(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(9)
  void *x, *fmt, *stats, *st;
  long long outer, inner;
  int32_t relu;
  uint64_t seed;
  adaption_qtensor xq, q;
  if (!tensor_ptr(a[0], &x) || (a[1] != Py_None && !qtensor(a[1], &xq)) || !i64(a[2], &outer) || !i64(a[3], &inner) ||
      !truth(a[4], &relu) || !qtensor(a[5], &q) || !u64(a[6], &seed) || !tensor_ptr(a[7], &fmt) || !tensor_ptr(a[8], &stats) ||
      !current_stream(&st))
    return nullptr;
  CALL(p_adaption_lp_act_stochastic((const float*)x, a[1] == Py_None ? nullptr : &xq, (size_t)outer, (size_t)inner, relu, q,
                                    (const adaption_qfmt*)fmt, seed, (adaption_stats*)stats, st))
  return answer(rc, "adaption_lp_act_stochastic");
}

// x, d_hist
PyObject* bit_histogram(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(2)
  void *x, *h, *st;
  long long count;
  if (!tensor_ptr(a[0], &x) || !numel(a[0], &count) || !tensor_ptr(a[1], &h) || !current_stream(&st)) return nullptr;
  CALL(p_adaption_bit_histogram((const float*)x, (size_t)count, (uint64_t*)h, st))
  return answer(rc, "adaption_bit_histogram");
}

// x (QTensor), d_hist
PyObject* width_histogram(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(2)
  adaption_qtensor q;
  long long outer, inner;
  void *h, *st;
  if (!qtensor(a[0], &q) || !attr_i64(a[0], s_outer, &outer) || !attr_i64(a[0], s_inner, &inner) || !tensor_ptr(a[1], &h) ||
      !current_stream(&st))
    return nullptr;
  CALL(p_adaption_width_histogram(q, (size_t)outer, (size_t)inner, (uint64_t*)h, st))
  return answer(rc, "adaption_width_histogram");
}

// shape, x (QTensor), w (QTensor), algo
PyObject* conv_workspace(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(4)
  Buffer shape;
  long long xn, xf, wn, wf, cs;
  int32_t algo;
  if (!shape.get(a[0], sizeof(adaption_conv_shape), "shape") || !attr_i64(a[1], s_n_bits, &xn) ||
      !attr_i64(a[1], s_frac_bits, &xf) || !attr_i64(a[1], s_c_stride, &cs) || !attr_i64(a[2], s_n_bits, &wn) ||
      !attr_i64(a[2], s_frac_bits, &wf) || !i32(a[3], &algo))
    return nullptr;
  const adaption_qfmt fx{(int32_t)xn, (int32_t)xf}, fw{(int32_t)wn, (int32_t)wf};
  return PyLong_FromSize_t(p_adaption_lp_conv_workspace_bytes((const adaption_conv_shape*)shape.b.buf, fx, fw, cs, algo));
}

// shape, x, w, y (QTensors), algo
PyObject* conv_pool_workspace(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(5)
  Buffer shape;
  long long xn, xf, wn, wf, yn, yf, cs, ycs;
  int32_t algo;
  if (!shape.get(a[0], sizeof(adaption_conv_shape), "shape") || !attr_i64(a[1], s_n_bits, &xn) ||
      !attr_i64(a[1], s_frac_bits, &xf) || !attr_i64(a[1], s_c_stride, &cs) || !attr_i64(a[2], s_n_bits, &wn) ||
      !attr_i64(a[2], s_frac_bits, &wf) || !attr_i64(a[3], s_n_bits, &yn) || !attr_i64(a[3], s_frac_bits, &yf) ||
      !attr_i64(a[3], s_c_stride, &ycs) || !i32(a[4], &algo))
    return nullptr;
  const adaption_qfmt fx{(int32_t)xn, (int32_t)xf}, fw{(int32_t)wn, (int32_t)wf}, fy{(int32_t)yn, (int32_t)yf};
  return PyLong_FromSize_t(
      p_adaption_lp_conv_pool_workspace_bytes((const adaption_conv_shape*)shape.b.buf, fx, fw, fy, cs, ycs, algo));
}

// B, K, O, x, w (QTensors), algo
PyObject* ip_workspace(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(6)
  long long B, K, O, xn, xf, wn, wf;
  int32_t algo;
  if (!i64(a[0], &B) || !i64(a[1], &K) || !i64(a[2], &O) || !attr_i64(a[3], s_n_bits, &xn) || !attr_i64(a[3], s_frac_bits, &xf) ||
      !attr_i64(a[4], s_n_bits, &wn) || !attr_i64(a[4], s_frac_bits, &wf) || !i32(a[5], &algo))
    return nullptr;
  const adaption_qfmt fx{(int32_t)xn, (int32_t)xf}, fw{(int32_t)wn, (int32_t)wf};
  return PyLong_FromSize_t(p_adaption_lp_ip_workspace_bytes(B, K, O, fx, fw, algo));
}

// shape, x, w, bias_q, bias_frac_bits, relu, mode, algo, y or None, d_stats, workspace
PyObject* conv_fwd(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(11)
  Buffer shape;
  adaption_qtensor x, w, y{};
  void *bias, *stats, *ws, *st;
  size_t wsb;
  int32_t bf, relu, mode, algo;
  if (!shape.get(a[0], sizeof(adaption_conv_shape), "shape") || !qtensor(a[1], &x) || !qtensor(a[2], &w) ||
      !tensor_ptr(a[3], &bias) || !i32(a[4], &bf) || !truth(a[5], &relu) || !i32(a[6], &mode) || !i32(a[7], &algo) ||
      (a[8] != Py_None && !qtensor(a[8], &y)) || !tensor_ptr(a[9], &stats) || !workspace(a[10], &ws, &wsb) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_lp_conv_fwd((const adaption_conv_shape*)shape.b.buf, x, w, (const int16_t*)bias, bf, relu, mode, algo, y,
                              (adaption_stats*)stats, ws, wsb, st))
  return answer(rc, "adaption_lp_conv_fwd");
}

// shape, x, w, bias_q, bias_frac_bits, relu, algo, y, seed, d_stats, workspace
PyObject* conv_fwd_stochastic(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(11)
  Buffer shape;
  adaption_qtensor x, w, y;
  void *bias, *stats, *ws, *st;
  size_t wsb;
  int32_t bf, relu, algo;
  uint64_t seed;
  if (!shape.get(a[0], sizeof(adaption_conv_shape), "shape") || !qtensor(a[1], &x) || !qtensor(a[2], &w) ||
      !tensor_ptr(a[3], &bias) || !i32(a[4], &bf) || !truth(a[5], &relu) || !i32(a[6], &algo) || !qtensor(a[7], &y) ||
      !u64(a[8], &seed) || !tensor_ptr(a[9], &stats) || !workspace(a[10], &ws, &wsb) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_lp_conv_fwd_stochastic((const adaption_conv_shape*)shape.b.buf, x, w, (const int16_t*)bias, bf, relu, algo, y,
                                         seed, (adaption_stats*)stats, ws, wsb, st))
  return answer(rc, "adaption_lp_conv_fwd_stochastic");
}

// shape, x, w, bias_q, bias_frac_bits, relu, algo, y, d_stats, workspace, phases
PyObject* conv_pool_fwd(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(11)
  Buffer shape;
  adaption_qtensor x, w, y;
  void *bias, *stats, *ws, *st;
  size_t wsb;
  int32_t bf, relu, algo, phases;
  if (!shape.get(a[0], sizeof(adaption_conv_shape), "shape") || !qtensor(a[1], &x) || !qtensor(a[2], &w) ||
      !tensor_ptr(a[3], &bias) || !i32(a[4], &bf) || !truth(a[5], &relu) || !i32(a[6], &algo) || !qtensor(a[7], &y) ||
      !tensor_ptr(a[8], &stats) || !workspace(a[9], &ws, &wsb) || !i32(a[10], &phases) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_lp_conv_pool_fwd((const adaption_conv_shape*)shape.b.buf, x, w, (const int16_t*)bias, bf, relu, algo, phases,
                                   y, (adaption_stats*)stats, ws, wsb, st))
  return answer(rc, "adaption_lp_conv_pool_fwd");
}

// B, K, O, x, w, bias_q, bias_frac_bits, relu, mode, algo, y or None, d_stats, workspace
PyObject* ip_fwd(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(13)
  adaption_qtensor x, w, y{};
  void *bias, *stats, *ws, *st;
  size_t wsb;
  long long B, K, O;
  int32_t bf, relu, mode, algo;
  if (!i64(a[0], &B) || !i64(a[1], &K) || !i64(a[2], &O) || !qtensor(a[3], &x) || !qtensor(a[4], &w) || !tensor_ptr(a[5], &bias) ||
      !i32(a[6], &bf) || !truth(a[7], &relu) || !i32(a[8], &mode) || !i32(a[9], &algo) || (a[10] != Py_None && !qtensor(a[10], &y)) ||
      !tensor_ptr(a[11], &stats) || !workspace(a[12], &ws, &wsb) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_lp_ip_fwd(B, K, O, x, w, (const int16_t*)bias, bf, relu, mode, algo, y, (adaption_stats*)stats, ws, wsb, st))
  return answer(rc, "adaption_lp_ip_fwd");
}

// B, K, O, x, w, bias_q, bias_frac_bits, relu, algo, y, seed, d_stats, workspace
PyObject* ip_fwd_stochastic(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(13)
  adaption_qtensor x, w, y;
  void *bias, *stats, *ws, *st;
  size_t wsb;
  long long B, K, O;
  int32_t bf, relu, algo;
  uint64_t seed;
  if (!i64(a[0], &B) || !i64(a[1], &K) || !i64(a[2], &O) || !qtensor(a[3], &x) || !qtensor(a[4], &w) || !tensor_ptr(a[5], &bias) ||
      !i32(a[6], &bf) || !truth(a[7], &relu) || !i32(a[8], &algo) || !qtensor(a[9], &y) || !u64(a[10], &seed) ||
      !tensor_ptr(a[11], &stats) || !workspace(a[12], &ws, &wsb) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_lp_ip_fwd_stochastic(B, K, O, x, w, (const int16_t*)bias, bf, relu, algo, y, seed, (adaption_stats*)stats, ws,
                                       wsb, st))
  return answer(rc, "adaption_lp_ip_fwd_stochastic");
}

// B, K, O, x, w, bias_q, bias_frac_bits, relu, mode, algo, y or None, d_stats
PyObject* ip_fwd_static_ws(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(12)
  adaption_qtensor x, w, y{};
  void *bias, *stats, *st;
  long long B, K, O;
  int32_t bf, relu, mode, algo;
  if (!i64(a[0], &B) || !i64(a[1], &K) || !i64(a[2], &O) || !qtensor(a[3], &x) || !qtensor(a[4], &w) || !tensor_ptr(a[5], &bias) ||
      !i32(a[6], &bf) || !truth(a[7], &relu) || !i32(a[8], &mode) || !i32(a[9], &algo) || (a[10] != Py_None && !qtensor(a[10], &y)) ||
      !tensor_ptr(a[11], &stats) || !current_stream(&st))
    return nullptr;
  CALL(p_adaption_lp_ip_fwd_static_ws(B, K, O, x, w, (const int16_t*)bias, bf, relu, mode, algo, y, (adaption_stats*)stats, st))
  return answer(rc, "adaption_lp_ip_fwd_static_ws");
}

// x, N, H, W, C, y
PyObject* maxpool(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(6)
  adaption_qtensor x, y;
  int32_t N, H, W, C;
  void* st;
  if (!qtensor(a[0], &x) || !i32(a[1], &N) || !i32(a[2], &H) || !i32(a[3], &W) || !i32(a[4], &C) || !qtensor(a[5], &y) ||
      !current_stream(&st))
    return nullptr;
  CALL(p_adaption_maxpool2x2(x, N, H, W, C, y, st))
  return answer(rc, "adaption_maxpool2x2");
}

// library path, AdaptionError, current device, stream of device
PyObject* bind(PyObject*, PyObject* const* a, Py_ssize_t nargs) {
  ARGS(4)
  const char* path = PyUnicode_AsUTF8(a[0]);
  if (path == nullptr) return nullptr;
  void* lib = dlopen(path, RTLD_NOW | RTLD_LOCAL);
  if (lib == nullptr) {
    PyErr_Format(PyExc_RuntimeError, "%s cannot be opened: %s", path, dlerror());
    return nullptr;
  }
#define RESOLVE(f)                                                        \
  p_##f = reinterpret_cast<decltype(p_##f)>(dlsym(lib, #f));              \
  if (p_##f == nullptr) {                                                 \
    PyErr_SetString(PyExc_RuntimeError, "the library lacks " #f);         \
    return nullptr;                                                       \
  }
  ADAPTION_FUNCTIONS(RESOLVE)
#undef RESOLVE
  for (int k = 1; k < 4; ++k) Py_INCREF(a[k]);
  Py_XSETREF(g_error, a[1]);
  Py_XSETREF(g_device, a[2]);
  Py_XSETREF(g_stream, a[3]);
  Py_RETURN_NONE;
}

#define METHOD(f) {#f, (PyCFunction)(void (*)(void))f, METH_FASTCALL, nullptr}
PyMethodDef methods[] = {METHOD(bind), METHOD(measure_range), METHOD(quantize), METHOD(fill_items), METHOD(quantize_batch),
                         METHOD(quantize_batch_stochastic), METHOD(quantize_stochastic), METHOD(lp_act),
                         METHOD(lp_act_stochastic), METHOD(bit_histogram), METHOD(width_histogram), METHOD(conv_workspace),
                         METHOD(conv_pool_workspace), METHOD(ip_workspace), METHOD(conv_fwd), METHOD(conv_fwd_stochastic),
                         METHOD(conv_pool_fwd), METHOD(ip_fwd), METHOD(ip_fwd_stochastic), METHOD(ip_fwd_static_ws),
                         METHOD(maxpool), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_adaption_native", "Argument marshalling of the C ABI.", -1, methods,
                      nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__adaption_native() {
  struct { PyObject** o; const char* s; } names[] = {
      {&s_lo, "lo"}, {&s_hi, "hi"}, {&s_q16, "q16"}, {&s_n_bits, "n_bits"}, {&s_frac_bits, "frac_bits"},
      {&s_c_stride, "c_stride"}, {&s_outer, "outer"}, {&s_inner, "inner"}, {&s_data_ptr, "data_ptr"}, {&s_numel, "numel"},
      {&s_itemsize, "itemsize"}};
  for (auto& n : names) {
    *n.o = PyUnicode_InternFromString(n.s);
    if (*n.o == nullptr) return nullptr;
  }
  return PyModule_Create(&module);
}
