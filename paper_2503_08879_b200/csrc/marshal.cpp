// The argument marshalling of binding.py's hot calls, in C.
//
// A hot call takes a handful of tensors, turns each into a pointer, one or two into strides, finds the current stream
// and calls the C interface.  Through ctypes that was 7 us of a decode call's 11.6 (a stream object built to be asked
// for its handle 3.4, the pointer and stride objects 2.3, the conversion of eleven arguments 0.9): more than the kernel of
// a short cache takes.  With this module the whole call takes 4.6.  Nothing is computed or kept: every call
// reads its arguments anew (any object with data_ptr(), integers with __index__, ctypes.ArgumentError for what is none).
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include "sagekv.h"

namespace {

typedef int (*ScoreFn)(sagekv_ctx *, const void *, const void *, sagekv_strides, int64_t, int32_t, int32_t, float *, int64_t, void *);
typedef int (*SelectFn)(sagekv_ctx *, const float *, int64_t, const void *, const void *, sagekv_strides, int64_t, int32_t, int32_t,
                        int32_t, int32_t *, void *, void *, sagekv_strides, sagekv_cache_state *, void *);
typedef int (*DecodeFn)(sagekv_ctx *, const void *, const void *, const void *, void *, void *, sagekv_strides,
                        const sagekv_cache_state *, void *, float *, void *);
typedef int (*PoolFn)(sagekv_ctx *, const float *, int64_t, int64_t, int32_t, int32_t, float *, int64_t, void *);
typedef int (*BoundsFn)(sagekv_ctx *, const void *, const void *, const void *, int64_t, float *, int64_t, void *);
typedef int (*TopkFn)(sagekv_ctx *, const float *, int64_t, int64_t, int32_t, int32_t *, void *);

ScoreFn g_score;
SelectFn g_select;
DecodeFn g_decode;
PoolFn g_pool;
BoundsFn g_bounds;
TopkFn g_topk;
PyObject *g_stream_of;   // callable: handle of the current stream of the current device, as an integer
PyObject *g_arg_error;   // ctypes.ArgumentError
PyObject *g_data_ptr, *g_stride;

// All of these return false with a Python exception set.
bool pointer(PyObject *t, void **out) {
  *out = nullptr;
  if (t == Py_None) return true;
  PyObject *v = PyObject_CallMethodNoArgs(t, g_data_ptr);
  if (v == nullptr) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return PyErr_Occurred() == nullptr;
}

bool integer(PyObject *o, int64_t *out) {
  *out = (int64_t)PyLong_AsUnsignedLongLongMask(o);   // as ctypes: no range check
  if (*out == -1 && PyErr_Occurred() != nullptr) {
    PyErr_Clear();
    PyErr_Format(g_arg_error, "'%.100s' object cannot be interpreted as an integer", Py_TYPE(o)->tp_name);
    return false;
  }
  return true;
}
bool integer(PyObject *o, int32_t *out) {
  int64_t v;
  if (!integer(o, &v)) return false;
  *out = (int32_t)(uint32_t)(uint64_t)v;
  return true;
}

// strides of a [B, H_kv, tokens, 128] tensor whose last dimension is contiguous
bool strides(PyObject *t, sagekv_strides *out) {
  PyObject *v = PyObject_CallMethodNoArgs(t, g_stride);
  if (v == nullptr) return false;
  int64_t s[4] = {0, 0, 0, 0};
  const bool four = PyTuple_Check(v) && PyTuple_GET_SIZE(v) == 4;
  for (int i = 0; four && i < 4; ++i) s[i] = PyLong_AsLongLong(PyTuple_GET_ITEM(v, i));
  Py_DECREF(v);
  if (PyErr_Occurred() != nullptr) return false;
  if (!four || s[3] != 1) {
    PyErr_SetString(PyExc_ValueError, "expected a [B, H_kv, tokens, head_dim] tensor with contiguous head_dim");
    return false;
  }
  out->batch_stride = s[0]; out->head_stride = s[1]; out->token_stride = s[2];
  return true;
}

// the context handle: a ctypes c_void_p, an integer or None
bool context(PyObject *o, sagekv_ctx **out) {
  *out = nullptr;
  if (o == Py_None) return true;
  if (PyLong_Check(o)) {
    *out = static_cast<sagekv_ctx *>(PyLong_AsVoidPtr(o));
    return PyErr_Occurred() == nullptr;
  }
  Py_buffer b;
  if (PyObject_GetBuffer(o, &b, PyBUF_SIMPLE) != 0) return false;
  const bool ok = b.len == (Py_ssize_t)sizeof(*out);
  if (ok) *out = *static_cast<sagekv_ctx **>(b.buf);
  PyBuffer_Release(&b);
  if (!ok) PyErr_SetString(g_arg_error, "not a context handle");
  return ok;
}

// the ctypes structure CacheState, held for the call
struct State {
  Py_buffer b{};
  sagekv_cache_state *p = nullptr;
  bool get(PyObject *o) {
    if (PyObject_GetBuffer(o, &b, PyBUF_WRITABLE) != 0) return false;
    if (b.len != (Py_ssize_t)sizeof(*p)) {
      PyErr_SetString(PyExc_TypeError, "expected a CacheState");
      return false;
    }
    p = static_cast<sagekv_cache_state *>(b.buf);
    return true;
  }
  ~State() { if (b.obj != nullptr) PyBuffer_Release(&b); }
};

bool current_stream(void **out) {
  PyObject *v = PyObject_CallNoArgs(g_stream_of);
  if (v == nullptr) return false;
  *out = PyLong_AsVoidPtr(v);
  Py_DECREF(v);
  return PyErr_Occurred() == nullptr;
}

bool count(Py_ssize_t n, Py_ssize_t want) {
  if (n != want) PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
  return n == want;
}

template <typename Call>
PyObject *answer(Call call) {
  int code;
  Py_BEGIN_ALLOW_THREADS
  code = call();
  Py_END_ALLOW_THREADS
  return PyLong_FromLong(code);
}

// ctx, q_last, K, n_ctx, n_init, n_recent, scores, scores_row_stride
PyObject *score(PyObject *, PyObject *const *a, Py_ssize_t n) {
  sagekv_ctx *ctx; void *q, *K, *scores, *stream; sagekv_strides ks; int64_t n_ctx, stride; int32_t n_init, n_recent;
  if (!count(n, 8) || !context(a[0], &ctx) || !pointer(a[1], &q) || !pointer(a[2], &K) || !strides(a[2], &ks) ||
      !integer(a[3], &n_ctx) || !integer(a[4], &n_init) || !integer(a[5], &n_recent) || !pointer(a[6], &scores) ||
      !integer(a[7], &stride) || !current_stream(&stream))
    return nullptr;
  return answer([&] { return g_score(ctx, q, K, ks, n_ctx, n_init, n_recent, static_cast<float *>(scores), stride, stream); });
}

// ctx, scores, scores_row_stride, K, V, n_ctx, n_init, n_recent, k, idx, Kc, Vc, state
PyObject *select_compact(PyObject *, PyObject *const *a, Py_ssize_t n) {
  sagekv_ctx *ctx; void *scores, *K, *V, *idx, *Kc, *Vc, *stream; sagekv_strides ks, cs;
  int64_t stride, n_ctx; int32_t n_init, n_recent, k; State st;
  if (!count(n, 13) || !context(a[0], &ctx) || !pointer(a[1], &scores) || !integer(a[2], &stride) || !pointer(a[3], &K) ||
      !pointer(a[4], &V) || !strides(a[3], &ks) || !integer(a[5], &n_ctx) || !integer(a[6], &n_init) ||
      !integer(a[7], &n_recent) || !integer(a[8], &k) || !pointer(a[9], &idx) || !pointer(a[10], &Kc) || !pointer(a[11], &Vc) ||
      !strides(a[10], &cs) || !st.get(a[12]) || !current_stream(&stream))
    return nullptr;
  return answer([&] {
    return g_select(ctx, static_cast<float *>(scores), stride, K, V, ks, n_ctx, n_init, n_recent, k, static_cast<int32_t *>(idx), Kc, Vc,
                    cs, st.p, stream);
  });
}

// ctx, q, k_new, v_new, Kc, Vc, state, out, lse
PyObject *decode_attn(PyObject *, PyObject *const *a, Py_ssize_t n) {
  sagekv_ctx *ctx; void *q, *kn, *vn, *Kc, *Vc, *out, *lse, *stream; sagekv_strides cs; State st;
  if (!count(n, 9) || !context(a[0], &ctx) || !pointer(a[1], &q) || !pointer(a[2], &kn) || !pointer(a[3], &vn) ||
      !pointer(a[4], &Kc) || !pointer(a[5], &Vc) || !strides(a[4], &cs) || !st.get(a[6]) || !pointer(a[7], &out) ||
      !pointer(a[8], &lse) || !current_stream(&stream))
    return nullptr;
  return answer([&] { return g_decode(ctx, q, kn, vn, Kc, Vc, cs, st.p, out, static_cast<float *>(lse), stream); });
}

// ctx, scores, scores_row_stride, n_ctx, n_init, n_recent, pooled, pooled_row_stride
PyObject *pool_scores(PyObject *, PyObject *const *a, Py_ssize_t n) {
  sagekv_ctx *ctx; void *scores, *pooled, *stream; int64_t stride, n_ctx, pooled_stride; int32_t n_init, n_recent;
  if (!count(n, 8) || !context(a[0], &ctx) || !pointer(a[1], &scores) || !integer(a[2], &stride) || !integer(a[3], &n_ctx) ||
      !integer(a[4], &n_init) || !integer(a[5], &n_recent) || !pointer(a[6], &pooled) || !integer(a[7], &pooled_stride) ||
      !current_stream(&stream))
    return nullptr;
  return answer([&] {
    return g_pool(ctx, static_cast<float *>(scores), stride, n_ctx, n_init, n_recent, static_cast<float *>(pooled), pooled_stride, stream);
  });
}

// ctx, q, kmin, kmax, n_blocks, bounds, bounds_row_stride
PyObject *quest_bounds(PyObject *, PyObject *const *a, Py_ssize_t n) {
  sagekv_ctx *ctx; void *q, *kmin, *kmax, *bounds, *stream; int64_t n_blocks, stride;
  if (!count(n, 7) || !context(a[0], &ctx) || !pointer(a[1], &q) || !pointer(a[2], &kmin) || !pointer(a[3], &kmax) ||
      !integer(a[4], &n_blocks) || !pointer(a[5], &bounds) || !integer(a[6], &stride) || !current_stream(&stream))
    return nullptr;
  return answer([&] { return g_bounds(ctx, q, kmin, kmax, n_blocks, static_cast<float *>(bounds), stride, stream); });
}

// ctx, scores, scores_row_stride, n, k_q, idx
PyObject *select_topk(PyObject *, PyObject *const *a, Py_ssize_t n) {
  sagekv_ctx *ctx; void *scores, *idx, *stream; int64_t stride, len; int32_t k_q;
  if (!count(n, 6) || !context(a[0], &ctx) || !pointer(a[1], &scores) || !integer(a[2], &stride) || !integer(a[3], &len) ||
      !integer(a[4], &k_q) || !pointer(a[5], &idx) || !current_stream(&stream))
    return nullptr;
  return answer([&] { return g_topk(ctx, static_cast<float *>(scores), stride, len, k_q, static_cast<int32_t *>(idx), stream); });
}

// addresses of the six entry points (score, select_compact, decode_attn, pool_scores, quest_bounds, select_topk), the
// callable that tells the current stream, ctypes.ArgumentError
PyObject *bind(PyObject *, PyObject *const *a, Py_ssize_t n) {
  if (!count(n, 8)) return nullptr;
  void *f[6];
  for (int i = 0; i < 6; ++i) {
    f[i] = PyLong_AsVoidPtr(a[i]);
    if (PyErr_Occurred() != nullptr) return nullptr;
  }
  g_score = reinterpret_cast<ScoreFn>(f[0]);
  g_select = reinterpret_cast<SelectFn>(f[1]);
  g_decode = reinterpret_cast<DecodeFn>(f[2]);
  g_pool = reinterpret_cast<PoolFn>(f[3]);
  g_bounds = reinterpret_cast<BoundsFn>(f[4]);
  g_topk = reinterpret_cast<TopkFn>(f[5]);
  Py_XSETREF(g_stream_of, Py_NewRef(a[6]));
  Py_XSETREF(g_arg_error, Py_NewRef(a[7]));
  Py_RETURN_NONE;
}

PyCFunction fast(PyObject *(*f)(PyObject *, PyObject *const *, Py_ssize_t)) {
  return reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f));
}

PyMethodDef g_methods[] = {
    {"bind", fast(bind), METH_FASTCALL, nullptr},
    {"score", fast(score), METH_FASTCALL, nullptr},
    {"select_compact", fast(select_compact), METH_FASTCALL, nullptr},
    {"decode_attn", fast(decode_attn), METH_FASTCALL, nullptr},
    {"pool_scores", fast(pool_scores), METH_FASTCALL, nullptr},
    {"quest_bounds", fast(quest_bounds), METH_FASTCALL, nullptr},
    {"select_topk", fast(select_topk), METH_FASTCALL, nullptr},
    {nullptr, nullptr, 0, nullptr}};

PyModuleDef g_module = {PyModuleDef_HEAD_INIT, "_marshal", nullptr, -1, g_methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__marshal(void) {
  g_data_ptr = PyUnicode_InternFromString("data_ptr");
  g_stride = PyUnicode_InternFromString("stride");
  if (g_data_ptr == nullptr || g_stride == nullptr) return nullptr;
  return PyModule_Create(&g_module);
}
