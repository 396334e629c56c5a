// binding.cpp -- Python entry points of libspade.so: checks of the torch tensors
// (type, device, layout, consistent shapes) and the call with their pointers and
// the stream.  Native because the checks of a dozen tensors and a 20-argument
// foreign call cost ~16 us from Python, as much as the GPU takes for a small
// verify step's kernel.  Every function takes its arguments by position and
// returns the library's status code; argument errors raise the Python exceptions.
#include <Python.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

#include "spade.h"

namespace {

using c10::ScalarType;

// Raised for an argument; the exception is set.
struct Bad {};

const char *type_name(ScalarType t) {
  switch (t) {
    case ScalarType::BFloat16: return "torch.bfloat16";
    case ScalarType::Float: return "torch.float32";
    case ScalarType::Int: return "torch.int32";
    default: return "torch.uint8";
  }
}

[[noreturn]] void value_error(const char *msg) {
  PyErr_SetString(PyExc_ValueError, msg);
  throw Bad{};
}

// A contiguous CUDA tensor of the given type (and rank, unless ndim < 0).
const at::Tensor &need(PyObject *o, const char *name, ScalarType type, int ndim) {
  if (o == Py_None) {
    PyErr_Format(PyExc_ValueError, "%s is required", name);
    throw Bad{};
  }
  const bool tensor = THPVariable_Check(o);
  if (!tensor || THPVariable_Unpack(o).scalar_type() != type) {
    PyObject *dt = PyObject_GetAttrString(o, "dtype");
    if (dt) {
      PyErr_Format(PyExc_TypeError, "%s must be %s, got %S", name, type_name(type), dt);
      Py_DECREF(dt);
    }
    throw Bad{};
  }
  const at::Tensor &t = THPVariable_Unpack(o);
  if (!t.is_cuda()) {
    PyErr_Format(PyExc_ValueError, "%s must be a CUDA tensor", name);
    throw Bad{};
  }
  if (!t.is_contiguous()) {
    PyErr_Format(PyExc_ValueError, "%s must be contiguous", name);
    throw Bad{};
  }
  if (ndim >= 0 && t.dim() != ndim) {
    PyErr_Format(PyExc_ValueError, "%s must have %d dims, got %ld", name, ndim, static_cast<long>(t.dim()));
    throw Bad{};
  }
  return t;
}

const at::Tensor &bf16(PyObject *o, const char *name, int ndim) { return need(o, name, ScalarType::BFloat16, ndim); }
const at::Tensor &f32(PyObject *o, const char *name, int ndim) { return need(o, name, ScalarType::Float, ndim); }
const at::Tensor &i32(PyObject *o, const char *name) { return need(o, name, ScalarType::Int, 1); }
const at::Tensor &u8(PyObject *o, const char *name) { return need(o, name, ScalarType::Byte, 1); }

const int32_t *ip(const at::Tensor &t) { return static_cast<const int32_t *>(t.data_ptr()); }
int32_t *ip_mut(const at::Tensor &t) { return static_cast<int32_t *>(t.data_ptr()); }
const float *fp(const at::Tensor *t) { return t ? static_cast<const float *>(t->data_ptr()) : nullptr; }
int32_t n32(int64_t v) { return static_cast<int32_t>(v); }

int32_t as_int(PyObject *o) {
  PyObject *n = PyNumber_Long(o);
  if (!n) throw Bad{};
  const long long v = PyLong_AsLongLong(n);
  Py_DECREF(n);
  if (v == -1 && PyErr_Occurred()) throw Bad{};
  return static_cast<int32_t>(v);
}
float as_float(PyObject *o) {
  const double v = PyFloat_AsDouble(o);
  if (v == -1.0 && PyErr_Occurred()) throw Bad{};
  return static_cast<float>(v);
}

// The given torch stream, or the current one of the current device.
spade_stream_t stream_of(PyObject *o) {
  if (o == Py_None) return reinterpret_cast<spade_stream_t>(c10::cuda::getCurrentCUDAStream().stream());
  PyObject *h = PyObject_GetAttrString(o, "cuda_stream");
  if (!h) throw Bad{};
  void *p = PyLong_AsVoidPtr(h);
  Py_DECREF(h);
  if (!p && PyErr_Occurred()) throw Bad{};
  return static_cast<spade_stream_t>(p);
}

// The library call runs without the interpreter lock (a launch may wait for
// room in the stream's queue).
struct NoGil {
  PyThreadState *state = PyEval_SaveThread();
  ~NoGil() { PyEval_RestoreThread(state); }
};

// Runs f, turning C++ exceptions into Python ones.
template <class F>
PyObject *guarded(Py_ssize_t n, Py_ssize_t want, F f) {
  if (n != want) {
    PyErr_Format(PyExc_TypeError, "expected %zd arguments, got %zd", want, n);
    return nullptr;
  }
  try {
    return PyLong_FromLong(static_cast<long>(f()));
  } catch (const Bad &) {
    return nullptr;
  } catch (const std::exception &e) {
    PyErr_SetString(PyExc_RuntimeError, e.what());
    return nullptr;
  }
}

struct Pools {
  const at::Tensor &k, &v, &table;
  int64_t num_pages, Hkv, page, D, max_pages;
};
Pools need_paged(PyObject *k_pool, PyObject *v_pool, PyObject *table) {
  const at::Tensor &k = bf16(k_pool, "k_pool", 4), &v = bf16(v_pool, "v_pool", 4);
  const at::Tensor &t = need(table, "block_table", ScalarType::Int, 2);
  if (v.sizes() != k.sizes()) value_error("k_pool and v_pool shapes differ");
  return Pools{k, v, t, k.size(0), k.size(1), k.size(2), k.size(3), t.size(1)};
}

// ---- attention -----------------------------------------------------------------------------
// q, k_cache, v_cache, ctx_lens, n_draft, cu_q, out, lse, max_k, workspace, status, stream
PyObject *attention(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 12, [&] {
    const at::Tensor &q = bf16(a[0], "q", 3), &k = bf16(a[1], "k_cache", 4), &v = bf16(a[2], "v_cache", 4);
    const at::Tensor &ctx = i32(a[3], "ctx_lens"), &nd = i32(a[4], "n_draft"), &cu = i32(a[5], "cu_q");
    const at::Tensor &st = i32(a[10], "status"), &out = bf16(a[6], "out", 3);
    void *lse = a[7] == Py_None ? nullptr : f32(a[7], "lse", 2).data_ptr();
    const at::Tensor &ws = u8(a[9], "workspace");
    if (v.sizes() != k.sizes()) value_error("k_cache and v_cache shapes differ");
    const int64_t R = q.size(0), Hq = q.size(1), D = q.size(2), B = k.size(0);
    if (k.size(3) != D || out.sizes() != q.sizes() || ctx.numel() != B || nd.numel() != B || cu.numel() != B + 1)
      value_error("inconsistent attention shapes");
    const spade_stream_t s = stream_of(a[11]);
    const int32_t max_k = as_int(a[8]);
    const NoGil released;
    return spade_verify_attention(q.data_ptr(), k.data_ptr(), v.data_ptr(), ip(ctx), ip(nd), ip(cu), out.data_ptr(),
                                  static_cast<float *>(lse), n32(B), n32(Hq), n32(k.size(1)), n32(D), n32(k.size(2)),
                                  max_k, n32(R), ws.data_ptr(), ws.numel(), ip_mut(st), s);
  });
}

// q, k_cache, v_cache, ctx_lens, n_draft, cu_q, out, lse, max_k, status, stream
PyObject *attention_noalloc(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 11, [&] {
    const at::Tensor &q = bf16(a[0], "q", -1), &k = bf16(a[1], "k_cache", -1), &v = bf16(a[2], "v_cache", -1);
    const at::Tensor &out = bf16(a[6], "out", -1);
    if (q.dim() != 3) value_error("q must have 3 dims");
    if (k.dim() != 4) value_error("k_cache must have 4 dims");
    const at::Tensor &ctx = i32(a[3], "ctx_lens"), &nd = i32(a[4], "n_draft"), &cu = i32(a[5], "cu_q");
    const at::Tensor &st = i32(a[9], "status");
    void *lse = a[7] == Py_None ? nullptr : f32(a[7], "lse", -1).data_ptr();
    const spade_stream_t s = stream_of(a[10]);
    const int32_t max_k = as_int(a[8]);
    const NoGil released;
    return spade_verify_attention_noalloc(q.data_ptr(), k.data_ptr(), v.data_ptr(), ip(ctx), ip(nd), ip(cu),
                                          out.data_ptr(), static_cast<float *>(lse), n32(k.size(0)), n32(q.size(1)),
                                          n32(k.size(1)), n32(q.size(2)), n32(k.size(2)), max_k, n32(q.size(0)),
                                          ip_mut(st), s);
  });
}

// q, k_pool, v_pool, block_table, ctx_lens, n_draft, cu_q, out, lse, max_k, workspace, status, stream
PyObject *attention_paged(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 13, [&] {
    const at::Tensor &q = bf16(a[0], "q", 3), &out = bf16(a[7], "out", 3);
    const Pools g = need_paged(a[1], a[2], a[3]);
    const at::Tensor &ctx = i32(a[4], "ctx_lens"), &nd = i32(a[5], "n_draft"), &cu = i32(a[6], "cu_q");
    const at::Tensor &st = i32(a[11], "status");
    void *lse = a[8] == Py_None ? nullptr : f32(a[8], "lse", 2).data_ptr();
    const at::Tensor &ws = u8(a[10], "workspace");
    const int64_t B = ctx.numel();
    if (q.size(2) != g.D || out.sizes() != q.sizes() || g.table.size(0) != B || nd.numel() != B || cu.numel() != B + 1)
      value_error("inconsistent paged attention shapes");
    const spade_stream_t s = stream_of(a[12]);
    const int32_t max_k = as_int(a[9]);
    const NoGil released;
    return spade_verify_attention_paged(q.data_ptr(), g.k.data_ptr(), g.v.data_ptr(), ip(g.table), ip(ctx), ip(nd),
                                        ip(cu), out.data_ptr(), static_cast<float *>(lse), n32(B), n32(q.size(1)),
                                        n32(g.Hkv), n32(g.D), n32(g.page), n32(g.num_pages), n32(g.max_pages),
                                        max_k, n32(q.size(0)), ws.data_ptr(), ws.numel(), ip_mut(st),
                                        s);
  });
}

// ---- LM head + accept ------------------------------------------------------------------------
// The ten leading arguments of every accept call: hidden, w_lm, draft_tokens,
// draft_probs, uniforms, mode, cu_q, n_draft, accepted_len, next_token.
struct Accept {
  const at::Tensor &hidden, &w, &uniforms, &tokens, &mode, &cu, &nd, &acc, &next;
  const at::Tensor *probs;
  int64_t B, R, H, V;
};
Accept accept_args(PyObject *const *a) {
  const at::Tensor &hidden = bf16(a[0], "hidden", 2), &w = bf16(a[1], "w_lm", 2), &u = f32(a[4], "uniforms", 1);
  const at::Tensor &tok = i32(a[2], "draft_tokens"), &mode = i32(a[5], "mode"), &cu = i32(a[6], "cu_q");
  const at::Tensor &nd = i32(a[7], "n_draft"), &acc = i32(a[8], "accepted_len"), &next = i32(a[9], "next_token");
  const at::Tensor *probs = a[3] == Py_None ? nullptr : &f32(a[3], "draft_probs", 2);
  return Accept{hidden, w, u, tok, mode, cu, nd, acc, next, probs, nd.numel(), hidden.size(0), hidden.size(1), w.size(0)};
}
bool accept_shapes(const Accept &c) {
  return c.w.size(1) == c.H && c.uniforms.numel() == c.R && c.tokens.numel() == c.R - c.B && c.cu.numel() == c.B + 1 &&
         c.mode.numel() == c.B && c.acc.numel() == c.B && c.next.numel() == c.B;
}
void probs_shape(const Accept &c) {
  if (c.probs && (c.probs->size(0) != c.R - c.B || c.probs->size(1) != c.V))
    value_error("draft_probs must be [R - B, V]");
}

// accept arguments, temperature, workspace, status, stream
PyObject *accept(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 14, [&] {
    const Accept c = accept_args(a);
    const at::Tensor &st = i32(a[12], "status"), &ws = u8(a[11], "workspace");
    if (!accept_shapes(c)) value_error("inconsistent accept shapes");
    probs_shape(c);
    if (a[10] == Py_None) {
      const spade_stream_t s = stream_of(a[13]);
      const NoGil released;
      return spade_verify_accept(c.hidden.data_ptr(), c.w.data_ptr(), ip(c.tokens), fp(c.probs), fp(&c.uniforms),
                                 ip(c.mode), ip(c.cu), ip(c.nd), ip_mut(c.acc), ip_mut(c.next), n32(c.B), n32(c.R),
                                 n32(c.H), n32(c.V), ws.data_ptr(), ws.numel(), ip_mut(st), s);
    }
    const at::Tensor &t = f32(a[10], "temperature", 1);
    if (t.numel() != c.B) value_error("temperature must be [B]");
    const spade_stream_t s = stream_of(a[13]);
    const NoGil released;
    return spade_verify_accept_temperature(c.hidden.data_ptr(), c.w.data_ptr(), ip(c.tokens), fp(c.probs),
                                           fp(&c.uniforms), ip(c.mode), fp(&t), ip(c.cu), ip(c.nd), ip_mut(c.acc),
                                           ip_mut(c.next), n32(c.B), n32(c.R), n32(c.H), n32(c.V), ws.data_ptr(),
                                           ws.numel(), ip_mut(st), s);
  });
}

// accept arguments, k_cache, v_cache, ctx_lens, workspace, status, stream
PyObject *accept_commit(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 16, [&] {
    const Accept c = accept_args(a);
    const at::Tensor &st = i32(a[14], "status"), &ctx = i32(a[12], "ctx_lens"), &ws = u8(a[13], "workspace");
    const at::Tensor &k = bf16(a[10], "k_cache", 4), &v = bf16(a[11], "v_cache", 4);
    if (!accept_shapes(c) || k.size(0) != c.B || v.sizes() != k.sizes() || ctx.numel() != c.B)
      value_error("inconsistent accept/commit shapes");
    probs_shape(c);
    const spade_stream_t s = stream_of(a[15]);
    const NoGil released;
    return spade_verify_accept_commit(c.hidden.data_ptr(), c.w.data_ptr(), ip(c.tokens), fp(c.probs), fp(&c.uniforms),
                                      ip(c.mode), ip(c.cu), ip(c.nd), ip_mut(c.acc), ip_mut(c.next), k.data_ptr(),
                                      v.data_ptr(), ip_mut(ctx), n32(c.B), n32(c.R), n32(c.H), n32(c.V), n32(k.size(1)),
                                      n32(k.size(3)), n32(k.size(2)), ws.data_ptr(), ws.numel(), ip_mut(st),
                                      s);
  });
}

// accept arguments, temperature, top_p, k_cache, v_cache, ctx_lens, workspace, status, stream
PyObject *accept_sampling(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 18, [&] {
    const Accept c = accept_args(a);
    const at::Tensor &st = i32(a[16], "status"), &ws = u8(a[15], "workspace");
    if (!accept_shapes(c)) value_error("inconsistent accept shapes");
    probs_shape(c);
    const at::Tensor *temp = nullptr, *top_p = nullptr;
    if (a[10] != Py_None) {
      temp = &f32(a[10], "temperature", 1);
      if (temp->numel() != c.B) value_error("temperature must be [B]");
    }
    if (a[11] != Py_None) {
      top_p = &f32(a[11], "top_p", 1);
      if (top_p->numel() != c.B) value_error("top_p must be [B]");
    }
    const bool commit = a[12] != Py_None;
    if (commit != (a[13] != Py_None) || commit != (a[14] != Py_None))
      value_error("give all of k_cache, v_cache, ctx_lens or none");
    void *kp = nullptr, *vp = nullptr;
    int32_t *cp = nullptr;
    int64_t Hkv = 0, D = 0, cap = 0;
    if (commit) {
      const at::Tensor &k = bf16(a[12], "k_cache", 4), &v = bf16(a[13], "v_cache", 4), &ctx = i32(a[14], "ctx_lens");
      if (k.size(0) != c.B || v.sizes() != k.sizes() || ctx.numel() != c.B) value_error("inconsistent cache shapes");
      kp = k.data_ptr();
      vp = v.data_ptr();
      cp = ip_mut(ctx);
      Hkv = k.size(1);
      cap = k.size(2);
      D = k.size(3);
    }
    const spade_stream_t s = stream_of(a[17]);
    const NoGil released;
    return spade_verify_accept_sampling(c.hidden.data_ptr(), c.w.data_ptr(), ip(c.tokens), fp(c.probs), fp(&c.uniforms),
                                        ip(c.mode), fp(temp), fp(top_p), ip(c.cu), ip(c.nd), ip_mut(c.acc),
                                        ip_mut(c.next), kp, vp, cp, n32(c.B), n32(c.R), n32(c.H), n32(c.V), n32(Hkv),
                                        n32(D), n32(cap), ws.data_ptr(), ws.numel(), ip_mut(st), s);
  });
}

// accept arguments, k_pool, v_pool, block_table, ctx_lens, workspace, status, stream
PyObject *accept_commit_paged(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 17, [&] {
    const Accept c = accept_args(a);
    const at::Tensor &st = i32(a[15], "status"), &ctx = i32(a[13], "ctx_lens"), &ws = u8(a[14], "workspace");
    const at::Tensor &k = bf16(a[10], "k_pool", 4), &v = bf16(a[11], "v_pool", 4);
    const at::Tensor &table = need(a[12], "block_table", ScalarType::Int, 2);
    if (!accept_shapes(c) || v.sizes() != k.sizes() || ctx.numel() != c.B || table.size(0) != c.B)
      value_error("inconsistent accept/commit shapes");
    probs_shape(c);
    const spade_stream_t s = stream_of(a[16]);
    const NoGil released;
    return spade_verify_accept_commit_paged(c.hidden.data_ptr(), c.w.data_ptr(), ip(c.tokens), fp(c.probs),
                                            fp(&c.uniforms), ip(c.mode), ip(c.cu), ip(c.nd), ip_mut(c.acc),
                                            ip_mut(c.next), k.data_ptr(), v.data_ptr(), ip(table), ip_mut(ctx), n32(c.B),
                                            n32(c.R), n32(c.H), n32(c.V), n32(k.size(1)), n32(k.size(3)), n32(k.size(2)),
                                            n32(k.size(0)), n32(table.size(1)), ws.data_ptr(), ws.numel(), ip_mut(st),
                                            s);
  });
}

// ---- QKV projection ----------------------------------------------------------------------------
// x, w_qkv, ctx_lens, n_draft, cu_q, q_out, k_cache, v_cache, Hq, Hkv, rope_theta, max_k, workspace, status, stream
PyObject *qkv(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 15, [&] {
    const at::Tensor &x = bf16(a[0], "x", 2), &w = bf16(a[1], "w_qkv", 2), &q = bf16(a[5], "q_out", 3);
    const at::Tensor &k = bf16(a[6], "k_cache", 4), &v = bf16(a[7], "v_cache", 4);
    const at::Tensor &ctx = i32(a[2], "ctx_lens"), &nd = i32(a[3], "n_draft"), &cu = i32(a[4], "cu_q");
    const at::Tensor &st = i32(a[13], "status");
    const int64_t R = x.size(0), H = x.size(1), B = k.size(0), D = k.size(3);
    const int32_t Hq = as_int(a[8]), Hkv = as_int(a[9]);
    if (k.size(1) != Hkv || v.sizes() != k.sizes() || q.size(0) != R || q.size(1) != Hq || q.size(2) != D ||
        w.size(0) != (Hq + 2 * static_cast<int64_t>(Hkv)) * D || w.size(1) != H || ctx.numel() != B ||
        nd.numel() != B || cu.numel() != B + 1)
      value_error("inconsistent qkv_rope shapes");
    const at::Tensor &ws = u8(a[12], "workspace");
    const spade_stream_t s = stream_of(a[14]);
    const int32_t max_k = as_int(a[11]);
    const float theta = as_float(a[10]);
    const NoGil released;
    return spade_verify_qkv_rope(x.data_ptr(), w.data_ptr(), ip(ctx), ip(nd), ip(cu), q.data_ptr(), k.data_ptr(),
                                 v.data_ptr(), n32(B), n32(R), n32(H), Hq, Hkv, n32(D), n32(k.size(2)), max_k,
                                 theta, ws.data_ptr(), ws.numel(), ip_mut(st), s);
  });
}

// x, w_qkv, block_table, ctx_lens, n_draft, cu_q, q_out, k_pool, v_pool, Hq, rope_theta, max_k, workspace, status, stream
PyObject *qkv_paged(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 15, [&] {
    const at::Tensor &x = bf16(a[0], "x", 2), &w = bf16(a[1], "w_qkv", 2), &q = bf16(a[6], "q_out", 3);
    const Pools g = need_paged(a[7], a[8], a[2]);
    const at::Tensor &ctx = i32(a[3], "ctx_lens"), &nd = i32(a[4], "n_draft"), &cu = i32(a[5], "cu_q");
    const at::Tensor &st = i32(a[13], "status");
    const int64_t R = x.size(0), H = x.size(1), B = ctx.numel();
    const int32_t Hq = as_int(a[9]);
    if (q.size(0) != R || q.size(1) != Hq || q.size(2) != g.D || w.size(0) != (Hq + 2 * g.Hkv) * g.D || w.size(1) != H ||
        g.table.size(0) != B || nd.numel() != B || cu.numel() != B + 1)
      value_error("inconsistent paged qkv_rope shapes");
    const at::Tensor &ws = u8(a[12], "workspace");
    const spade_stream_t s = stream_of(a[14]);
    const int32_t max_k = as_int(a[11]);
    const float theta = as_float(a[10]);
    const NoGil released;
    return spade_verify_qkv_rope_paged(x.data_ptr(), w.data_ptr(), ip(g.table), ip(ctx), ip(nd), ip(cu), q.data_ptr(),
                                       g.k.data_ptr(), g.v.data_ptr(), n32(B), n32(R), n32(H), Hq, n32(g.Hkv), n32(g.D),
                                       n32(g.page), n32(g.num_pages), n32(g.max_pages), max_k, theta,
                                       ws.data_ptr(), ws.numel(), ip_mut(st), s);
  });
}

// ---- KV commit ---------------------------------------------------------------------------------
// k_cache, v_cache, ctx_lens, accepted_len, n_draft, status, stream
PyObject *commit(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 7, [&] {
    const at::Tensor &k = bf16(a[0], "k_cache", 4), &v = bf16(a[1], "v_cache", 4), &ctx = i32(a[2], "ctx_lens");
    const at::Tensor &acc = i32(a[3], "accepted_len"), &nd = i32(a[4], "n_draft"), &st = i32(a[5], "status");
    const spade_stream_t s = stream_of(a[6]);
    const NoGil released;
    return spade_kv_commit(k.data_ptr(), v.data_ptr(), ip_mut(ctx), ip(acc), ip(nd), n32(k.size(0)), n32(k.size(1)),
                           n32(k.size(3)), n32(k.size(2)), ip_mut(st), s);
  });
}

// k_pool, v_pool, block_table, ctx_lens, accepted_len, n_draft, status, stream
PyObject *commit_paged(PyObject *, PyObject *const *a, Py_ssize_t n) {
  return guarded(n, 8, [&] {
    const Pools g = need_paged(a[0], a[1], a[2]);
    const at::Tensor &ctx = i32(a[3], "ctx_lens"), &acc = i32(a[4], "accepted_len"), &nd = i32(a[5], "n_draft");
    const at::Tensor &st = i32(a[6], "status");
    const int64_t B = ctx.numel();
    if (g.table.size(0) != B) value_error("block_table must have one row per sequence");
    const spade_stream_t s = stream_of(a[7]);
    const NoGil released;
    return spade_kv_commit_paged(g.k.data_ptr(), g.v.data_ptr(), ip(g.table), ip_mut(ctx), ip(acc), ip(nd), n32(B),
                                 n32(g.Hkv), n32(g.D), n32(g.page), n32(g.num_pages), n32(g.max_pages), ip_mut(st),
                                 s);
  });
}

#define ENTRY(f) {#f, reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(f)), METH_FASTCALL, nullptr}
PyMethodDef methods[] = {
    ENTRY(attention), ENTRY(attention_noalloc), ENTRY(attention_paged), ENTRY(accept), ENTRY(accept_commit),
    ENTRY(accept_sampling), ENTRY(accept_commit_paged), ENTRY(qkv), ENTRY(qkv_paged), ENTRY(commit),
    ENTRY(commit_paged), {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_spade_native", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__spade_native() { return PyModule_Create(&module); }
