// qkv_common.cuh -- what the two forms of the verify block's QKV projection share:
// the output side (rotary angle, where a head's slice of a row goes), the row
// table and the launch of the cluster form.
#pragma once
#include <cuda_bf16.h>

#include <cstdint>

#include "internal.h"
#include "ptx.cuh"

namespace spade {
namespace qkv {

constexpr int kKChunk = 64;  // k elements per 128-byte swizzled row

// The call's outputs and sequences.
struct Call {
  const int32_t *ctx_lens;
  const int32_t *n_draft;
  const int32_t *cu_q;
  __nv_bfloat16 *q_out;    // [R, Hq, D]
  __nv_bfloat16 *k_cache;  // [B, Hkv, cap, D] (or a pool, see block_table)
  __nv_bfloat16 *v_cache;
  int32_t *status;
  int B, R, H, Hq, Hkv, D, cap, max_k;
  float inv_freq[64];  // theta^(-2j/D), j < D/2, rounded from double on the host
  // Paged caches (block_table null: dense [B, Hkv, cap, D]): pools
  // [num_pages, Hkv, page_size, D], block_table [B, max_pages].
  const int32_t *block_table;
  int page_size, max_pages, num_pages;
};

// Sine and cosine of pos * f: the product as an exact pair (a + e == pos * f),
// reduced to [-pi, pi] with 2 pi split in two parts (Cody and Waite's method),
// then the SFU's sine and cosine (accurate to a few 1e-7 on that interval).
__device__ __forceinline__ void rope_angle(int pos, float f, float *sn, float *cs) {
  const float x = static_cast<float>(pos);  // exact: positions are below 2^24
  const float a = x * f;
  const float e = fmaf(x, f, -a);
  const float k = rintf(a * 0.15915494309189535f);           // 1 / (2 pi)
  float r = fmaf(-k, 6.28318548202514648f, a);               // 2 pi rounded to float
  r = fmaf(-k, -1.7484555314695172e-07f, r);                 // 2 pi minus that
  __sincosf(r + e, sn, cs);
}

// Row table (thread et of nt, `bar` a barrier among them): position of every
// verify row and its row in the caches, at KV head 0 (32 bits: 2^32 rows of the
// smallest head are 550 GB); rows of invalid sequences are marked kNoRow, and
// CTA 0 reports them.  (Looked up as the rows are stored, pages and divisions
// made up a third of the epilogue at 389 paged rows.)
constexpr uint32_t kNoRow = 0xffffffffu;
template <class Bar>
__device__ __forceinline__ void build_rows(const Call &p, uint32_t *s_row, int32_t *s_rpos, int et, int nt, Bar bar) {
  for (int r = et; r < p.R; r += nt) s_row[r] = kNoRow;
  bar();
  for (int b = et; b < p.B; b += nt) {
    const int c = p.ctx_lens[b], k = p.n_draft[b];
    const int q0 = p.cu_q[b], q1 = p.cu_q[b + 1];
    int bad = 0;
    if (c < 0 || k < 0 || k > p.max_k || q0 < 0 || q1 > p.R || q1 - q0 != k + 1) bad = SPADE_DEV_BAD_INDEX;
    else if (static_cast<int64_t>(c) + k + 1 > p.cap) bad = SPADE_DEV_CAPACITY;
    if (!bad && p.block_table) {
      // Every page the block writes must exist.
      for (int i = 0; i <= k; ++i) {
        const int pg = p.block_table[static_cast<int64_t>(b) * p.max_pages + (c + i) / p.page_size];
        if (pg < 0 || pg >= p.num_pages) bad = SPADE_DEV_BAD_INDEX;
      }
    }
    if (bad) {
      if (blockIdx.x == 0) atomicOr(p.status, bad);
      continue;
    }
    for (int i = 0; i <= k; ++i) {
      const int pos = c + i;
      if (p.block_table) {
        const uint32_t pg = p.block_table[static_cast<int64_t>(b) * p.max_pages + pos / p.page_size];
        s_row[q0 + i] = pg * p.Hkv * p.page_size + pos % p.page_size;
      } else {
        s_row[q0 + i] = static_cast<uint32_t>(b) * p.Hkv * p.cap + pos;
      }
      s_rpos[q0 + i] = pos;
    }
  }
  bar();
}

// Where outputs go, copied from the call once (in a function that is not
// inlined the compiler would reload the parameters after every store).
struct OutMap {
  __nv_bfloat16 *q_out, *k_cache, *v_cache;
  int Hq, Hkv, D;
  int head_rows;  // cache rows from one KV head to the next
};
__device__ __forceinline__ OutMap out_map(const Call &c) {
  return OutMap{c.q_out, c.k_cache, c.v_cache, c.Hq, c.Hkv, c.D, c.block_table ? c.page_size : c.cap};
}

// Four consecutive rotary pairs (j0 .. j0 + 3 with j0 + D/2 ..; y1, y2) of head hg
// (among the Hq + 2 Hkv of the projection) of verify row r: rotation of query and
// key pairs and the bf16 stores, to q_out or the row's cache row (see
// build_rows).  4 bf16 = 8 bytes at each half (j0 a multiple of
// 4, rows 16-byte aligned).
__device__ __forceinline__ void store_quad(const OutMap &p, const float *s_freq, uint32_t row, int r, int pos, int hg, int j0,
                                           float (&y1)[4], float (&y2)[4]) {
  const int half = p.D / 2;
  if (hg < p.Hq + p.Hkv) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      float sn, cs;
      rope_angle(pos, s_freq[j0 + e], &sn, &cs);
      const float o1 = y1[e] * cs - y2[e] * sn, o2 = y2[e] * cs + y1[e] * sn;
      y1[e] = o1;
      y2[e] = o2;
    }
  }
  __nv_bfloat16 *dst;
  if (hg < p.Hq) {
    dst = p.q_out + (static_cast<size_t>(r) * p.Hq + hg) * p.D;
  } else {
    const int hk = hg < p.Hq + p.Hkv ? hg - p.Hq : hg - p.Hq - p.Hkv;
    __nv_bfloat16 *cache = hg < p.Hq + p.Hkv ? p.k_cache : p.v_cache;
    dst = cache + (static_cast<size_t>(row) + static_cast<uint32_t>(hk) * p.head_rows) * p.D;
  }
  *reinterpret_cast<uint2 *>(dst + j0) = make_uint2(pack_bf16(y1[0], y1[1]), pack_bf16(y1[2], y1[3]));
  *reinterpret_cast<uint2 *>(dst + j0 + half) = make_uint2(pack_bf16(y2[0], y2[1]), pack_bf16(y2[2], y2[3]));
}

// Cluster form (qkv_cluster.cu).  Whether it takes these sizes on `sms` SMs, and
// its launch (x [R, H], w_qkv [(Hq + 2 Hkv) D, H]).
bool cluster_fits(const Call &c, int sms);
spade_status launch_cluster(const Call &c, const void *x, const void *w_qkv, int sms, cudaStream_t stream);

}  // namespace qkv
}  // namespace spade
