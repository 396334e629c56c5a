// accept_common.cuh -- what the one-launch LM head (verify_accept.cu) and the
// two-launch one (lm_head_pairs.cu, accept_rows.cu) share: the call's
// parameters, the statistics epilogue of a 128-entry vocabulary tile, and the
// rows phase -- merge of the slice statistics, accept tests (Sec. III-C),
// nucleus, KV commit and the draw of the correction / bonus token -- that
// follows once every slice of the vocabulary is done.
#pragma once
#include <cuda_bf16.h>

#include <cfloat>
#include <climits>
#include <cstddef>
#include <cstdint>

#include "internal.h"
#include "ptx.cuh"

namespace spade {
namespace accept {

constexpr int kTileV = 128;    // vocab rows per tile and SM (MMA M, or half of a pair's M)
constexpr int kKChunk = 64;    // K elements per 128-byte swizzle row
constexpr int kEpiWarps = 8;   // two per tensor-memory lane quarter
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kWarps = 2 + kEpiWarps;
constexpr int kThreads = 32 * kWarps;
constexpr int kMaxRes = 256;   // verify rows of the one-launch path (MMA N <= 256)
constexpr int kMaxR = 512;     // verify rows per call
constexpr int kMaxB = 256;
constexpr int kMaxNC = 256;    // CTAs (vocabulary slices) per launch
constexpr int kMaxGroup = 32;  // CTAs that draw one sequence's token together
constexpr int kMinShare = 2048;  // vocabulary entries that make one more CTA in a group worth its barrier
constexpr int kTmemCols = 512;
constexpr int kSmemMax = 227 * 1024;                // shared memory a CTA may have
constexpr int kWChunkBytes = kTileV * kKChunk * 2;  // 16 KB: one tile x one k-chunk
constexpr int kBlk = 16;       // verify rows per statistics block
constexpr int kTStride = kBlk + 1;
constexpr int kTBufBytes = kEpiWarps * 32 * kTStride * 4;  // the warps' transpose buffers
constexpr float kLog2e = 1.4426950408889634f;

// One accept call: inputs, outputs and workspace.
struct Call {
  const int32_t *draft_tokens;
  const float *draft_probs;
  const float *uniforms;
  const int32_t *mode;
  const int32_t *cu_q;
  const int32_t *n_draft;
  int32_t *accepted_len;
  int32_t *next_token;
  int32_t *status;
  const float *temperature;  // [B] softmax temperature of each sequence, or null (all 1)
  const float *top_p;        // [B] nucleus mass of each sequence, or null (no truncation)
  unsigned *bar;     // barrier words (kBarBytes), zero between calls but for generations
  float4 *pstat;     // [R][NC]: slice max, slice sum-exp, slice argmax (bits), -
  float *ldraft;     // [R]: logit of the row's draft token
  float4 *gstat;     // [R]: merged row max, sum-exp, argmax (bits), accept bit
  float *logits;     // [R][ldl]: logits of the rows of sampled sequences (before temperature)
  float2 *zpart;     // [2 attempts][B][kMaxGroup]: share masses of the sampled distribution (float-float)
  unsigned *nhist;   // [2][kMaxGroup][R][kNucBins]: bin masses of the nucleus search (2^31 = all of p)
  // Fused KV commit (null kc: not requested): clear the rejected draft slots of
  // the caches [B, Hkv, cap, Dk] and advance ctx_lens once the decisions exist.
  uint4 *kc, *vc;
  int32_t *ctx_lens;
  int Hkv, Dk, cap;
  // Paged caches (block_table non-null): kc / vc are pools [num_pages, Hkv,
  // page_size, Dk]; slot s of sequence b is row s % page_size of page
  // block_table[b * max_pages + s / page_size]; cap = max_pages * page_size.
  const int32_t *block_table;
  int page_size, max_pages, num_pages;
  int B, R, V;
  int NC;    // vocabulary slices (CTAs of the statistics phase)
  int ldl;   // floats per logits row, a multiple of 4
  int qvec;  // draft_probs rows may be read as float4 (16-byte aligned rows)
};

// bar.sync is the aligned form: every lane of a warp must arrive together.
// Lanes that ran ahead of a divergent lane (a lane-0-only loop) reconverge
// first, so no warp reaches the barrier before all of its lanes do.
__device__ __forceinline__ void named_bar(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void block_sync() {
  __syncwarp();
  __syncthreads();
}

__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Barrier words: the grid barrier's arrival count at word 0 and its generation
// in kReplicas copies, a 128-byte line each (CTA c polls copy c % kReplicas:
// 152 CTAs polling one line queue on it); then one (count, generation) pair of
// lines per group of CTAs that draws a token together.
constexpr int kReplicas = 8;
constexpr int kGenWord = 32;
constexpr int kGroupWord = 512;
constexpr int kBarBytes = kGroupWord * 4 + kMaxNC * 2 * kGenWord * 4;
static_assert(kGenWord * (kReplicas + 1) <= kGroupWord, "grid barrier words fit their region");
constexpr int kNucBinBits = 5;                 // key bits decided per round of the nucleus search
constexpr int kNucBins = 1 << kNucBinBits;     // bins per round
constexpr int kNucRounds = 4;                  // all 20 key bits, see nuc_key
constexpr int kNucSubs = 2;                    // independent bin copies per lane
static_assert(kNucBins == 32, "one lane per bin");

// Merge of (max, sum of exp(x - max), argmax) summaries; lowest index wins ties.
__device__ __forceinline__ void stat_merge(float &m, float &s, int &i, float om, float os, int oi) {
  const float M = fmaxf(m, om);
  if (M == -INFINITY) {
    s = 0.f;
  } else {
    s = s * ex2((m - M) * kLog2e) + os * ex2((om - M) * kLog2e);
  }
  if (om > m || (om == m && oi < i)) i = oi;
  m = M;
}

// 1 / T for sequence b: p = softmax(l / T).  A temperature that is not
// positive and finite is reported and taken as 1.
__device__ __forceinline__ float inv_temp(const Call &p, int b) {
  if (p.temperature == nullptr || b < 0) return 1.f;
  const float t = __ldg(p.temperature + b);
  if (!(t > 0.f) || !(t < INFINITY)) {
    atomicOr(p.status, SPADE_DEV_BAD_INDEX);
    return 1.f;
  }
  return 1.f / t;
}

// Top-p (nucleus) threshold search over the scaled logits l of a row.  The
// nucleus is S = {x : l_x >= tau}, tau the largest logit value whose upper
// mass F(tau) = sum_{l_x >= tau} p_x reaches top_p (tokens tied with the
// boundary are in).  The search runs on integer keys
//   L(l) = floor((l - base) * 2^15),  base = m - 31.5  (m: the row maximum),
// a monotone map of l onto [0, 2^20) for every l >= base (p below base is at
// most V e^-31.5); each of kNucRounds rounds fixes 5 more bits of the key of
// the boundary, keeping the highest bin whose upper mass still reaches top_p.
// The nucleus is then {x : L(l_x) >= L_tau}: the same key decides the bins,
// the accept test and the sampling, so all three agree bit for bit.  Logits
// within one key step (2^-15 = 3.1e-5 in l) are not told apart.
constexpr float kNucSpan = 31.5f;
constexpr int kNucKeyBits = 20;
constexpr float kNucScale = 32768.f;  // key steps per unit of l
// y = fma(l, 2^15, -base 2^15) equals (l - base) rounded, times 2^15 (scaling
// by a power of two commutes with rounding); adding 2^23 rounded toward -inf
// leaves floor(y) in the low mantissa bits for 0 <= y < 2^23 (no conversion
// instruction), and a negative key for y < 0.  Monotone in l throughout.
// nb65 = -base * 2^15 (exact).  nuc_key_bits is the float's bit pattern,
// 0x4B000000 + L for L >= 0 (the constant's low 24 bits are zero, so shifts
// of the pattern and of L differ by a constant).
constexpr int kNucKeyBias = 0x4B000000;
__device__ __forceinline__ int nuc_key_bits(float l, float nb65) {
  return __float_as_int(__fadd_rd(__fmaf_rn(l, kNucScale, nb65), 8388608.f));
}
__device__ __forceinline__ int nuc_key(float l, float base) {
  return nuc_key_bits(l, -kNucScale * base) - kNucKeyBias;
}
// top_p of sequence b when it truncates p (0 < top_p < 1), else 1.
__device__ __forceinline__ float seq_top_p(const Call &p, int b) {
  if (p.top_p == nullptr || b < 0) return 1.f;
  const float t = __ldg(p.top_p + b);
  return (t > 0.f && t < 1.f) ? t : 1.f;
}

// Float-float numbers (hi + lo, about 48 significant bits) for the sums that
// place u*Z: GB300's fp64 rate is a small fraction of fp32, so the cumulative
// masses use error-free fp32 transformations instead of doubles.
struct ff2 {
  float hi, lo;
};
// Knuth's TwoSum: s + e == a + b exactly.
__device__ __forceinline__ ff2 two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  const float e = (a - (s - bb)) + (b - bb);
  return ff2{s, e};
}
__device__ __forceinline__ ff2 ff_norm(float hi, float lo) {
  const float s = hi + lo;
  return ff2{s, lo - (s - hi)};
}
__device__ __forceinline__ ff2 ff_add(ff2 a, ff2 b) {
  const ff2 s = two_sum(a.hi, b.hi);
  return ff_norm(s.hi, s.lo + a.lo + b.lo);
}
__device__ __forceinline__ ff2 ff_add_f(ff2 a, float b) {
  const ff2 s = two_sum(a.hi, b);
  return ff_norm(s.hi, s.lo + a.lo);
}
__device__ __forceinline__ ff2 ff_sub(ff2 a, ff2 b) { return ff_add(a, ff2{-b.hi, -b.lo}); }
// a * b with the product's rounding error recovered by an fma.
__device__ __forceinline__ ff2 ff_mul_f(ff2 a, float b) {
  const float p = a.hi * b;
  float e = fmaf(a.hi, b, -p);
  e = fmaf(a.lo, b, e);
  return ff_norm(p, e);
}
__device__ __forceinline__ bool ff_gt(ff2 a, ff2 b) {
  const ff2 d = ff_sub(a, b);
  return d.hi > 0.f || (d.hi == 0.f && d.lo > 0.f);
}
__device__ __forceinline__ ff2 ff_shfl(ff2 v, int src) {
  return ff2{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}
__device__ __forceinline__ ff2 warp_sum_ff(ff2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = ff_add(v, ff2{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)});
  return ff_shfl(v, 0);  // one value for every lane
}
// Inclusive prefix sum over the warp's lanes.
__device__ __forceinline__ ff2 warp_scan_ff(ff2 v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const ff2 t{__shfl_up_sync(0xffffffffu, v.hi, o), __shfl_up_sync(0xffffffffu, v.lo, o)};
    if (lane >= o) v = ff_add(t, v);
  }
  return v;
}

// Arrival at a barrier of n CTAs (one thread, after a CTA barrier that orders
// the CTA's writes before it): the last arrival resets the count and bumps the
// generation words.  Returns the generation seen before arriving; *last: this
// arrival completed the barrier and there is nothing to wait for.
__device__ __forceinline__ unsigned bar_arrive(unsigned *count, unsigned *gen, int copies, int my_copy, int n,
                                               bool *last) {
  const unsigned seen = ld_relaxed(gen + kGenWord * my_copy);  // before arriving (the release orders it first)
  unsigned arrived;
  asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(arrived) : "l"(count) : "memory");
  *last = arrived == static_cast<unsigned>(n) - 1;
  if (*last) {
    asm volatile("st.relaxed.gpu.global.u32 [%0], 0;" ::"l"(count) : "memory");
    // One release fence orders everything above before all the copies.
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    for (int r = 0; r < copies; ++r)
      asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(gen + kGenWord * r) : "memory");
  }
  return seen;
}
// Bounded poll for a generation newer than `seen` (one thread).
__device__ __forceinline__ bool bar_poll(const unsigned *gen_p, unsigned seen) {
  bool ok = true;
  const uint64_t t0 = globaltimer();
  while (ld_relaxed(gen_p) == seen) {
    if (globaltimer() - t0 > kWaitLimitNs) { ok = false; break; }
    __nanosleep(20);
  }
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  return ok;
}

// Device-wide barrier among the nctas co-resident CTAs (cooperative launch).
// Returns false if the wait expired.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, int nctas) {
  __shared__ int s_ok;
  block_sync();
  if (threadIdx.x == 0) {
    bool last;
    const int copy = blockIdx.x % kReplicas;
    const unsigned seen = bar_arrive(bar, bar + kGenWord, kReplicas, copy, nctas, &last);
    s_ok = last || bar_poll(bar + kGenWord * (1 + copy), seen);
  }
  block_sync();
  return s_ok != 0;
}

// Row range and mode of sequence b.
struct SeqInfo {
  int r0, k;    // first row, drafts
  bool valid;   // consistent with cu_q, its rows and drafts inside the call's
  bool stoch;   // sampled: stochastic, with q for its drafts (none needed without drafts)
};
__device__ __forceinline__ SeqInfo seq_info(const Call &p, int b) {
  SeqInfo q;
  const int r1 = p.cu_q[b + 1];
  q.r0 = p.cu_q[b];
  q.k = p.n_draft[b];
  q.valid = q.r0 >= 0 && q.k >= 0 && r1 <= p.R && r1 > q.r0 && r1 - q.r0 - 1 == q.k &&
            (q.k == 0 || (q.r0 >= b && q.r0 - b + q.k <= p.R - p.B));
  q.stoch = q.valid && p.mode[b] == 1 && (p.draft_probs != nullptr || q.k == 0);
  return q;
}

// Per-row tables of the statistics epilogue (the epilogue warps, thread et of
// kEpiThreads, while the first stages already stream): draft token (-1: none), 1 / T, and which rows' logits
// are kept for the draw (bit n % 16 of word n / 16).  Row n = cu_q[b] + i is
// position i of sequence b; it holds draft i for i < k_b.  nrows: a multiple
// of 16 that covers the rows.
__device__ __forceinline__ void setup_rows(const Call &p, int nrows, int32_t *s_draft, float *s_it, unsigned *s_keep,
                                           int et) {
  for (int n = et; n < nrows; n += kEpiThreads) { s_draft[n] = -1; s_it[n] = 1.f; }
  for (int w = et; w < nrows / kBlk; w += kEpiThreads) s_keep[w] = 0u;
  named_bar(1, kEpiThreads);
  for (int b = et; b < p.B; b += kEpiThreads) {
    const SeqInfo q = seq_info(p, b);
    if (!q.valid) {
      atomicOr(p.status, SPADE_DEV_BAD_INDEX);
      continue;
    }
    const float it = inv_temp(p, b);
    for (int i = 0; i <= q.k; ++i) {
      const int n = q.r0 + i;
      s_it[n] = it;
      if (i < q.k) s_draft[n] = p.draft_tokens[n - b];
      if (q.stoch) atomicOr(&s_keep[n / kBlk], 1u << (n % kBlk));
    }
  }
  named_bar(1, kEpiThreads);
}

// Running statistics of a block's 16 rows over the entries one warp has seen:
// maxima, sums of exp(x - maximum) and argmaxima.
struct BlkStat {
  float m[kBlk], s[kBlk];
  int i[kBlk];
};
__device__ __forceinline__ void blk_init(BlkStat &st, int lane) {
  if (lane < kBlk) {
    st.m[lane] = -INFINITY;
    st.s[lane] = 0.f;
    st.i[lane] = INT_MAX;
  }
}

// Statistics of 16 verify rows (r0 ..) over one warp's 32 vocabulary entries
// (v0 + lane), read from the 16 accumulator columns at `taddr`.  A 32 x 17
// shared-memory transpose gives lane (row = lane % 16, half = lane / 16) one
// row over 16 entries, reduced serially; the two halves meet by a shuffle each
// for the maximum and the sum.  The argmax search runs only when the block
// raises a row's running maximum.  Rows whose bit is set in `keep` also store
// their logits, 128 contiguous bytes per row and warp.
__device__ __forceinline__ void stat_block(const Call &p, uint32_t taddr, int r0, int v0, int v_hi, unsigned keep,
                                           const int32_t *s_draft, const float *s_it, float *T, int lane, BlkStat &st) {
  uint32_t raw[kBlk];
  tmem_ld8(taddr, raw);
  tmem_ld8(taddr + 8, raw + 8);
  tmem_wait_ld();
  const bool mine = v0 + lane < v_hi;  // lanes past the slice are masked
  if (keep != 0u) {
    float *dst = p.logits + static_cast<size_t>(r0) * p.ldl + v0 + lane;
#pragma unroll
    for (int r = 0; r < kBlk; ++r)
      if ((keep >> r) & 1u) {
        if (mine) dst[static_cast<size_t>(r) * p.ldl] = __uint_as_float(raw[r]);
      }
  }
#pragma unroll
  for (int r = 0; r < kBlk; ++r) T[lane * kTStride + r] = mine ? __uint_as_float(raw[r]) : -INFINITY;
  __syncwarp();
  const int row = lane % kBlk, vb = (lane / kBlk) * kBlk;  // 16 entries from v0 + vb on
  const int n = r0 + row;
  const float it = s_it[n];  // logits at the row's temperature, l / T
  const float rm = st.m[row];
  float x[kBlk];
  float m = -INFINITY;
#pragma unroll
  for (int i = 0; i < kBlk; ++i) {
    x[i] = __fmul_rn(T[(vb + i) * kTStride + row], it);
    m = fmaxf(m, x[i]);
  }
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, kBlk));
  const float M = fmaxf(rm, m);
  float a0 = 0.f, a1 = 0.f;
  if (M != -INFINITY) {
#pragma unroll
    for (int i = 0; i < kBlk; i += 2) {
      a0 += ex2((x[i] - M) * kLog2e);
      a1 += ex2((x[i + 1] - M) * kLog2e);
    }
  }
  a0 += a1;
  a0 += __shfl_xor_sync(0xffffffffu, a0, kBlk);
  const bool raised = m > rm;
  int idx = INT_MAX;
  if (__any_sync(0xffffffffu, raised)) {
#pragma unroll
    for (int i = kBlk - 1; i >= 0; --i)
      if (x[i] == m) idx = v0 + vb + i;
    idx = min(idx, __shfl_xor_sync(0xffffffffu, idx, kBlk));  // the lowest index of the maximum
  }
  if (lane < kBlk && M != -INFINITY) {
    st.s[row] = st.s[row] * ex2((rm - M) * kLog2e) + a0;
    if (raised) {
      st.m[row] = m;
      st.i[row] = idx;
    }
  }
  const int d = s_draft[n] - (v0 + vb);
  if (d >= 0 && d < kBlk && v0 + vb + d < v_hi) p.ldraft[n] = __fmul_rn(T[(vb + d) * kTStride + row], it);
  __syncwarp();
}

// Merge of the epilogue warps' statistics ([kEpiWarps][nblk], written and
// synchronised by the caller) into this CTA's slice partials.
__device__ __forceinline__ void publish_slice(const Call &p, const BlkStat *stats, int nblk, int c, int et) {
  for (int n = et; n < p.R; n += kEpiThreads) {
    float m = -INFINITY, s = 0.f;
    int idx = INT_MAX;
#pragma unroll
    for (int w = 0; w < kEpiWarps; ++w) {
      const BlkStat &st = stats[w * nblk + n / kBlk];
      stat_merge(m, s, idx, st.m[n % kBlk], st.s[n % kBlk], st.i[n % kBlk]);
    }
    __stcg(&p.pstat[static_cast<size_t>(n) * p.NC + c], make_float4(m, s, __int_as_float(idx), 0.f));
  }
}

// Shared memory of the rows phase.
struct RowsSmem {
  int n_st, n_gr, first, nl, owner, owner_warp, last, retry;
  unsigned gen;
  int abort;
  ff2 tgt, wtgt;
  ff2 wm[kWarps];        // masses of the warps' parts of this CTA's share
  int st[kMaxB];         // sampled sequences, ascending
  int gr[kMaxB];         // greedy and invalid ones
  float m[kMaxR], z[kMaxR];           // rows of the sequence at hand: maximum, sum of exponentials
  float u[kMaxR], q[kMaxR], l[kMaxR]; // uniform, q(draft), draft logit
  int arg[kMaxR], d[kMaxR], ok[kMaxR];
  int tkey[kMaxR];       // nucleus key threshold (INT_MIN: all of p)
  // Nucleus search only (one-launch path, at most 256 rows):
  int npre[kMaxRes];
  unsigned nab[kMaxRes];
  unsigned hist[kMaxRes][kNucBins];
  float bins[kWarps][kNucSubs * kNucBins * 32];
};
constexpr size_t kRowsBytesPlain = offsetof(RowsSmem, npre);

// Barrier of the gs CTAs of group g, split so that work that needs no other
// CTA can run between the two halves.
__device__ __forceinline__ void group_arrive(const Call &p, RowsSmem &s, int g, int gs) {
  block_sync();
  if (gs > 1 && threadIdx.x == 0) {
    unsigned *count = p.bar + kGroupWord + g * 2 * kGenWord;
    bool last;
    s.gen = bar_arrive(count, count + kGenWord, 1, 0, gs, &last);
    s.last = last;
  }
}
__device__ __forceinline__ void group_wait(const Call &p, RowsSmem &s, int g, int gs) {
  if (gs > 1 && threadIdx.x == 0 && !s.last && !s.abort &&
      !bar_poll(p.bar + kGroupWord + g * 2 * kGenWord + kGenWord, s.gen)) {
    atomicOr(p.status, SPADE_DEV_TIMEOUT);
    s.abort = 1;
  }
  block_sync();
}

// Merged statistics and accept bits of the rows of sequence b, one warp per
// row over the NC slice partials.  Greedy: the draft is the argmax (lowest
// index on ties); stochastic: u < p(d) / q(d) (Sec. III-C).
__device__ __forceinline__ void decide_rows(const Call &p, RowsSmem &s, int b, const SeqInfo &q, bool writer, int warp,
                                            int lane) {
  constexpr int kLoads = kMaxNC / 32;
#pragma unroll 1
  for (int i = warp; i <= q.k; i += kWarps) {
    const int n = q.r0 + i;
    float4 part[kLoads];
#pragma unroll
    for (int j = 0; j < kLoads; ++j) {
      const int cc = j * 32 + lane;
      part[j] = cc < p.NC ? __ldcg(&p.pstat[static_cast<size_t>(n) * p.NC + cc])
                          : make_float4(-INFINITY, 0.f, __int_as_float(INT_MAX), 0.f);
    }
    int d = -1;
    float u = 0.f, qd = 0.f, ld = 0.f;
    if (i < q.k) {
      d = p.draft_tokens[n - b];
      u = p.uniforms[n];
      if (d >= 0 && d < p.V) {
        ld = __ldcg(&p.ldraft[n]);
        if (q.stoch) qd = __ldg(&p.draft_probs[static_cast<size_t>(n - b) * p.V + d]);
      }
    }
    float m = -INFINITY, z = 0.f;
    int idx = INT_MAX;
#pragma unroll
    for (int j = 0; j < kLoads; ++j) stat_merge(m, z, idx, part[j].x, part[j].y, __float_as_int(part[j].z));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, m, o);
      const float oz = __shfl_xor_sync(0xffffffffu, z, o);
      const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
      stat_merge(m, z, idx, om, oz, oi);
    }
    if (lane == 0) {  // lane 0's values are everyone's
      int ok = 0;
      if (i < q.k) {
        if (d < 0 || d >= p.V) {
          atomicOr(p.status, SPADE_DEV_BAD_INDEX);
        } else if (!q.stoch) {
          ok = d == idx;
        } else {
          const float pd = expf(ld - m) / z;
          ok = (qd > 0.f) ? (u < pd / qd) : (pd > 0.f);
        }
      }
      s.m[i] = m;
      s.z[i] = z;
      s.arg[i] = idx;
      s.ok[i] = ok;
      s.d[i] = d;
      s.u[i] = u;
      s.q[i] = qd;
      s.l[i] = ld;
      s.tkey[i] = INT_MIN;
      if (writer) __stcg(&p.gstat[n], make_float4(m, z, __int_as_float(idx), __int_as_float(ok)));
    }
  }
  block_sync();
}

// Index of the first rejected draft among rows [0, upto), else upto.
__device__ __forceinline__ int first_reject(RowsSmem &s, int upto, int tid) {
  if (tid == 0) s.first = upto;
  block_sync();
  for (int i = tid; i < upto; i += kThreads)
    if (!s.ok[i]) atomicMin(&s.first, i);
  block_sync();
  return s.first;
}

// KV commit of sequence b (Algorithm 1 context update), by one CTA: slots
// [0, ctx_b + a] stay, the rejected drafts' slots [ctx_b + a + 1, ctx_b + k]
// are cleared and ctx_lens[b] advances by a + 1.
__device__ __forceinline__ void commit_seq(const Call &p, int b, int k, int a, int tid) {
  const int ctx = p.ctx_lens[b];
  int bad_page = 0;
  const bool fits = ctx >= 0 && static_cast<int64_t>(ctx) + k + 1 <= p.cap;
  const int lo = ctx + a + 1;
  const int32_t *bt = p.block_table ? p.block_table + static_cast<int64_t>(b) * p.max_pages : nullptr;
  if (bt && fits) {
    // Every page the rejected slots use must exist before anything is cleared.
    for (int j = tid; j < k - a; j += kThreads) {
      const int pg = bt[(lo + j) / p.page_size];
      bad_page |= pg < 0 || pg >= p.num_pages;
    }
  }
  __syncwarp();
  bad_page = __syncthreads_or(bad_page);  // every thread has read ctx_lens[b] before it changes
  if (!fits || bad_page) {
    if (tid == 0) atomicOr(p.status, fits || ctx < 0 ? SPADE_DEV_BAD_INDEX : SPADE_DEV_CAPACITY);
    return;
  }
  const int vec = p.Dk / 8;  // 16-byte vectors per slot
  const int per_head = (k - a) * vec;
  const int total = p.Hkv * per_head;
  const uint4 zero = make_uint4(0, 0, 0, 0);
  for (int e = tid; e < total; e += kThreads) {
    const int h = e / per_head;
    const int r = e - h * per_head;
    size_t off;
    if (bt) {
      const int slot = lo + r / vec;
      off = ((static_cast<size_t>(bt[slot / p.page_size]) * p.Hkv + h) * p.page_size + slot % p.page_size) * vec +
            r % vec;
    } else {
      off = ((static_cast<size_t>(b) * p.Hkv + h) * p.cap + lo) * vec + r;
    }
    p.kc[off] = zero;
    p.vc[off] = zero;
  }
  if (tid == 0) p.ctx_lens[b] = lo;
}

// This CTA's share [lo, hi) of the vocabulary in a group of gs, shares a
// multiple of 4 entries (logits rows are read as float4).
__device__ __forceinline__ void share_of(int V, int gs, int rank, int *lo, int *hi) {
  const int per = ((V + gs - 1) / gs + 3) & ~3;
  *lo = min(V, rank * per);
  *hi = min(V, *lo + per);
}

// Top-p: the nucleus of the rows of sequence b that can decide anything (see
// nuc_key), its group together.  A draft row whose u is past p(d) / (top_p q(d))
// is rejected whatever its nucleus (the nucleus holds at least top_p of p), so
// the rows after the first such row are not searched.  Per round every CTA bins
// its share of each row -- lane-private fp32 bins in kNucSubs copies (lane i's
// words all in bank i: no conflicts, no shared-memory atomics per value), summed
// in a fixed order and added to the row's bins in fixed point (2^31 = all of p:
// integer sums, the same in any order) -- publishes them, and after the group
// barrier sums every CTA's bins itself, so a round takes one barrier.  Two
// buffers alternate: a CTA writes a round's bins only after every CTA has read
// those of two rounds before.
__device__ __forceinline__ void nucleus(const Call &p, RowsSmem &s, int b, const SeqInfo &q, float top, int g,
                                        int rank, int gs, int lo, int hi, int tid, int warp, int lane) {
  if (tid == 0) s.nl = q.k + 1;
  block_sync();
  for (int i = tid; i < q.k; i += kThreads) {
    const bool in_range = s.d[i] >= 0 && s.d[i] < p.V;
    const float most = expf(s.l[i] - s.m[i]) / s.z[i] / top * 1.0001f;  // p(d) renormalised, at most
    if (!in_range || (s.q[i] > 0.f && s.u[i] >= most / s.q[i])) atomicMin(&s.nl, i + 1);
  }
  block_sync();
  const int nl = s.nl;
  for (int i = tid; i < nl; i += kThreads) {
    s.npre[i] = isfinite(s.m[i]) && s.z[i] > 0.f ? 0 : -1;  // -1: all of p
    s.nab[i] = 0u;
  }
  const float IT = inv_temp(p, b);
  const int parts = nl < kWarps ? kWarps / nl : 1;  // warps per row
  const int per = ((hi - lo + parts - 1) / parts + 127) & ~127;
  float *bins = s.bins[warp] + lane;
#pragma unroll 1
  for (int r = 0; r < kNucRounds; ++r) {
    const int sh = kNucKeyBits - kNucBinBits * (r + 1);  // this round's bin: key bits [sh, sh + 5)
    for (int e = tid; e < nl * kNucBins; e += kThreads) s.hist[e / kNucBins][e % kNucBins] = 0u;
    block_sync();
#pragma unroll 1
    for (int item = warp; item < nl * parts; item += kWarps) {
      const int i = item / parts, part = item - i * parts;
      const int pre = s.npre[i];
      if (pre < 0) continue;
      const float M = s.m[i];
      const float nb65 = -kNucScale * __fsub_rn(M, kNucSpan);
      const float mlog = -M * kLog2e;
      const int pre_bits = pre + (kNucKeyBias >> (sh + kNucBinBits));  // the range's key prefix, as bits
      const float *lg = p.logits + static_cast<size_t>(q.r0 + i) * p.ldl;
      const int plo = lo + part * per, phi = min(hi, plo + per);
#pragma unroll 8
      for (int k = 0; k < kNucSubs * kNucBins; ++k) bins[k * 32] = 0.f;
#pragma unroll 1
      for (int e0 = plo + 4 * lane; e0 < phi; e0 += 4 * 128) {
        float4 v4[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
          v4[j] = e0 + 128 * j < phi ? __ldcg(reinterpret_cast<const float4 *>(lg + e0 + 128 * j))
                                     : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float x[4] = {v4[j].x, v4[j].y, v4[j].z, v4[j].w};
          float ex[4];
          int a[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float l = __fmul_rn(x[c], IT);
            const int kbits = nuc_key_bits(l, nb65);
            const bool in = e0 + 128 * j + c < phi && (kbits >> (sh + kNucBinBits)) == pre_bits;
            ex[c] = in ? ex2(__fmaf_rn(l, kLog2e, mlog)) : 0.f;
            a[c] = ((c % kNucSubs) * kNucBins + ((kbits >> sh) & (kNucBins - 1))) * 32;
          }
#pragma unroll
          for (int c = 0; c < 4; c += kNucSubs) {
            float v[kNucSubs];
#pragma unroll
            for (int h = 0; h < kNucSubs; ++h) v[h] = bins[a[c + h]];
#pragma unroll
            for (int h = 0; h < kNucSubs; ++h) bins[a[c + h]] = v[h] + ex[c + h];
          }
        }
      }
      __syncwarp();
      // Lane = bin: its sum over the 32 lanes' copies, read along a diagonal.
      const float *all = s.bins[warp];
      float f = 0.f;
#pragma unroll 8
      for (int j = 0; j < 32; ++j)
#pragma unroll
        for (int h = 0; h < kNucSubs; ++h) f += all[(h * kNucBins + lane) * 32 + ((j + lane) & 31)];
      const unsigned fixed = __float2uint_rn(f * (0x1p31f / s.z[i]));
      if (fixed != 0u) atomicAdd(&s.hist[i][lane], fixed);
      __syncwarp();
    }
    block_sync();
    if (gs > 1) {
      unsigned *mine = p.nhist + (static_cast<size_t>((r & 1) * kMaxGroup + rank) * p.R + q.r0) * kNucBins;
      for (int e = tid; e < nl * kNucBins; e += kThreads) __stcg(&mine[e], s.hist[e / kNucBins][e % kNucBins]);
      group_arrive(p, s, g, gs);
      group_wait(p, s, g, gs);
    }
    // C_k = mass of keys at or above bin k plus the mass above the range: keep
    // the highest bin with C_k >= top_p.  Sums stay below 2^33.
#pragma unroll 1
    for (int i = warp; i < nl; i += kWarps) {
      unsigned long long own = 0;
      if (gs > 1) {
        const unsigned *src =
            p.nhist + (static_cast<size_t>((r & 1) * kMaxGroup) * p.R + q.r0 + i) * kNucBins + lane;
#pragma unroll 8
        for (int c = 0; c < gs; ++c) own += __ldcg(src + static_cast<size_t>(c) * p.R * kNucBins);
      } else {
        own = s.hist[i][lane];
      }
      unsigned long long C = own;  // suffix sum over lanes >= this one
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_down_sync(0xffffffffu, C, o);
        if (lane + o < 32) C += t;
      }
      C += s.nab[i];
      // top_p * 2^31 is exact in fp32; the target is its ceiling.
      const unsigned long long target = static_cast<unsigned long long>(ceilf(top * 0x1p31f));
      const unsigned ge = __ballot_sync(0xffffffffu, C >= target);
      const int kb = ge ? 31 - __clz(ge) : 0;  // C_k falls with k
      const unsigned long long ck = __shfl_sync(0xffffffffu, C, kb);
      const unsigned long long above = __shfl_sync(0xffffffffu, C - own, kb);
      if (lane == 0 && s.npre[i] >= 0) {
        s.npre[i] = (s.npre[i] << kNucBinBits) | kb;
        // The mass above the new prefix's range; after the last round F(tau).
        const unsigned long long F = r + 1 < kNucRounds ? above : ck;
        s.nab[i] = F > 0xffffffffull ? 0xffffffffu : static_cast<unsigned>(F);
      }
      __syncwarp();
    }
    block_sync();
  }
  // L_tau = the final prefix; p on S renormalised by S_nuc = F(tau).  The
  // accept tests are taken again under the nucleus.
  for (int i = tid; i < nl; i += kThreads) {
    const unsigned F = s.nab[i];
    if (s.npre[i] < 0 || F == 0u) continue;  // all of p
    const float S = s.z[i] * (static_cast<float>(F) * 0x1p-31f);
    const int tkey = s.npre[i] << (kNucKeyBits - kNucBinBits * kNucRounds);
    const float base = __fsub_rn(s.m[i], kNucSpan);
    s.tkey[i] = tkey;
    s.z[i] = S;
    if (i < q.k && s.d[i] >= 0 && s.d[i] < p.V) {
      const float pd = nuc_key(s.l[i], base) >= tkey ? expf(s.l[i] - s.m[i]) / S : 0.f;
      s.ok[i] = (s.q[i] > 0.f) ? (s.u[i] < pd / s.q[i]) : (pd > 0.f);
    }
  }
  block_sync();
}

// The distribution to draw from, entry by entry: max(0, p - q) or p.
struct Dist {
  const float *lg;  // logits row
  const float *q;   // draft distribution, or null: p
  float M, invS, IT, base;
  int tkey;
  bool qvec;
};
__device__ __forceinline__ void dist_load4(const Dist &t, int e, int hi, float4 &l4, float4 &q4) {
  l4 = __ldcg(reinterpret_cast<const float4 *>(t.lg + e));
  q4 = make_float4(0.f, 0.f, 0.f, 0.f);
  if (t.q) {
    if (t.qvec) {
      q4 = __ldg(reinterpret_cast<const float4 *>(t.q + e));
    } else {
      q4.x = __ldg(t.q + e);
      if (e + 1 < hi) q4.y = __ldg(t.q + e + 1);
      if (e + 2 < hi) q4.z = __ldg(t.q + e + 2);
      if (e + 3 < hi) q4.w = __ldg(t.q + e + 3);
    }
  }
}
__device__ __forceinline__ float dist_term(const Dist &t, float l, float q, bool in_share) {
  const float lv = __fmul_rn(l, t.IT);
  const bool in = t.tkey == INT_MIN || nuc_key(lv, t.base) >= t.tkey;
  const float pv = in ? ex2((lv - t.M) * kLog2e) * t.invS : 0.f;
  const float rv = t.q ? fmaxf(0.f, pv - q) : pv;
  return in_share ? rv : 0.f;
}
__device__ __forceinline__ void dist_terms(const Dist &t, int e, int hi, const float4 &l4, const float4 &q4,
                                           float (&x)[4]) {
  x[0] = dist_term(t, l4.x, q4.x, e < hi);
  x[1] = dist_term(t, l4.y, q4.y, e + 1 < hi);
  x[2] = dist_term(t, l4.z, q4.z, e + 2 < hi);
  x[3] = dist_term(t, l4.w, q4.w, e + 3 < hi);
}

// The draw of sequence b by its group: next_token[b] is the first entry whose
// cumulative mass exceeds u Z.  Terms are fp32, every sum float-float, so the
// cumulative masses that place u Z are as exact as the terms allow.  Each warp
// sums a contiguous part of the CTA's share; the shares' masses meet in the
// workspace, every CTA finds the owner of u Z from the same masses, and the
// owner's warp that holds it scans its part again.  A residual with no mass is
// retried on p (every CTA sees the same total, so all retry together).
// `commit`: the group's first CTA updates the cache while the masses travel.
__device__ __forceinline__ void draw_token(const Call &p, RowsSmem &s, int b, const SeqInfo &q, int a, int g, int rank,
                                           int gs, int lo, int hi, bool commit, int tid, int warp, int lane) {
  const int n = q.r0 + a;
  Dist t;
  t.lg = p.logits + static_cast<size_t>(n) * p.ldl;
  t.q = a < q.k ? p.draft_probs + static_cast<size_t>(n - b) * p.V : nullptr;
  t.M = s.m[a];
  t.invS = 1.f / s.z[a];
  t.IT = inv_temp(p, b);
  t.base = __fsub_rn(t.M, kNucSpan);
  t.tkey = s.tkey[a];
  t.qvec = p.qvec != 0;
  const float u = p.uniforms[q.r0 + q.k];
  const int per = ((hi - lo + kWarps - 1) / kWarps + 127) & ~127;  // entries per warp
  const int wlo = min(hi, lo + warp * per), whi = min(hi, wlo + per);
#pragma unroll 1
  for (int attempt = 0; attempt < 2; ++attempt) {
    float sh[4] = {0.f, 0.f, 0.f, 0.f}, sl[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int e0 = wlo + 4 * lane; e0 < whi; e0 += 4 * 128) {
      float4 l4[4], q4[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        l4[j] = q4[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e0 + 128 * j < whi) dist_load4(t, e0 + 128 * j, whi, l4[j], q4[j]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float x[4];
        dist_terms(t, e0 + 128 * j, whi, l4[j], q4[j], x);
        // Compensated chains: the terms are >= 0, so ordering the two addends
        // by size makes the error term exact.
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float sm = sh[c] + x[c];
          sl[c] += (fmaxf(sh[c], x[c]) - sm) + fminf(sh[c], x[c]);
          sh[c] = sm;
        }
      }
    }
    const ff2 mass = warp_sum_ff(ff_add(ff_add(ff_norm(sh[0], sl[0]), ff_norm(sh[1], sl[1])),
                                        ff_add(ff_norm(sh[2], sl[2]), ff_norm(sh[3], sl[3]))));
    if (lane == 0) s.wm[warp] = mass;
    block_sync();
    float2 *zp = p.zpart + (static_cast<size_t>(attempt) * p.B + b) * kMaxGroup;
    if (tid == 0) {
      ff2 z{0.f, 0.f};
      for (int w = 0; w < kWarps; ++w) z = ff_add(z, s.wm[w]);
      __stcg(&zp[rank], make_float2(z.hi, z.lo));
    }
    group_arrive(p, s, g, gs);
    if (attempt == 0 && commit && rank == 0) commit_seq(p, b, q.k, a, tid);
    group_wait(p, s, g, gs);
    if (warp == 0) {
      const float2 zz = lane < gs ? __ldcg(&zp[lane]) : make_float2(0.f, 0.f);
      const ff2 mine{zz.x, zz.y};
      const ff2 incl = warp_scan_ff(mine, lane);
      const ff2 tot = ff_shfl(incl, 31);
      const bool ok = tot.hi > 0.f && isfinite(tot.hi);
      const ff2 target = ff_mul_f(tot, u);
      const unsigned hit = __ballot_sync(0xffffffffu, ok && mine.hi > 0.f && ff_gt(incl, target));
      const unsigned pos = __ballot_sync(0xffffffffu, ok && mine.hi > 0.f);
      // Rounding past the total clamps to the last share with mass.
      const int own = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : -1);
      const ff2 before = ff_shfl(ff_sub(incl, mine), own < 0 ? 0 : own);
      if (lane == 0) {
        s.retry = !ok;
        s.owner = own;
        s.tgt = ff_sub(target, before);  // target left inside the owner's share
      }
    }
    block_sync();
    if (!s.retry) {
      if (attempt == 1 && rank == 0 && tid == 0) atomicOr(p.status, SPADE_DEV_FALLBACK);
      break;
    }
    t.q = nullptr;  // the residual has no mass: sample p
  }
  if (s.retry || s.owner < 0) {
    if (rank == 0 && tid == 0) p.next_token[b] = -1;  // p has no mass either
    return;
  }
  if (s.owner != rank) return;
  // The warp part holding the target, then the entry, in vocabulary order.
  if (warp == 0) {
    const ff2 mine = lane < kWarps ? s.wm[lane] : ff2{0.f, 0.f};
    const ff2 incl = warp_scan_ff(mine, lane);
    const unsigned hit = __ballot_sync(0xffffffffu, mine.hi > 0.f && ff_gt(incl, s.tgt));
    const unsigned pos = __ballot_sync(0xffffffffu, mine.hi > 0.f);
    const int own = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
    const ff2 before = ff_shfl(ff_sub(incl, mine), own);
    if (lane == 0) {
      s.owner_warp = own;
      s.wtgt = hit ? ff_sub(s.tgt, before) : ff2{INFINITY, 0.f};  // rounding: clamp to the last mass
    }
  }
  block_sync();
  if (warp == s.owner_warp) {
    const ff2 target = s.wtgt;
    ff2 run{0.f, 0.f};
    int found = -1, last = -1;  // last: the last entry with mass so far
#pragma unroll 1
    for (int e0 = wlo; e0 < whi && found < 0; e0 += 128) {
      const int e = e0 + 4 * lane;
      float4 l4 = make_float4(0.f, 0.f, 0.f, 0.f), q4 = l4;
      if (e < whi) dist_load4(t, e, whi, l4, q4);
      float x[4];
      dist_terms(t, e, whi, l4, q4, x);
      ff2 mine{x[0], 0.f};
#pragma unroll
      for (int c = 1; c < 4; ++c) mine = ff_add_f(mine, x[c]);
      const ff2 incl = ff_add(run, warp_scan_ff(mine, lane));
      const unsigned hit = __ballot_sync(0xffffffffu, mine.hi > 0.f && ff_gt(incl, target));
      const unsigned pos = __ballot_sync(0xffffffffu, mine.hi > 0.f);
      const int src = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : -1);
      if (src >= 0) {
        // Lane src's first entry past the target, else its last one with mass.
        ff2 acc = ff_sub(incl, mine);
        int at = -1;
        bool over = false;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          acc = ff_add_f(acc, x[c]);
          if (x[c] > 0.f && !over) {
            at = e + c;
            over = hit != 0u && ff_gt(acc, target);
          }
        }
        at = __shfl_sync(0xffffffffu, at, src);
        if (hit) found = at;
        else last = at;
      }
      run = ff_shfl(incl, 31);
    }
    if (lane == 0) p.next_token[b] = found >= 0 ? found : (last >= 0 ? last : wlo);
  }
}

// After the statistics of every slice (a grid barrier, or the previous launch's
// end): decisions, outputs, commit and the draws.  Sampled sequences are dealt
// to groups of CTAs from the front of the grid, greedy ones to single CTAs
// from its end; no group waits for another.
__device__ __forceinline__ void rows_phase(const Call &p, RowsSmem &s, int c, int nctas) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    int ns = 0, ng = 0;
    for (int b0 = 0; b0 < p.B; b0 += 32) {
      const int b = b0 + lane;
      const bool st = b < p.B && seq_info(p, b).stoch;
      const unsigned ms = __ballot_sync(0xffffffffu, st);
      const unsigned mg = __ballot_sync(0xffffffffu, b < p.B && !st);
      const unsigned below = (1u << lane) - 1u;
      if (st) s.st[ns + __popc(ms & below)] = b;
      else if (b < p.B) s.gr[ng + __popc(mg & below)] = b;
      ns += __popc(ms);
      ng += __popc(mg);
    }
    if (lane == 0) {
      s.n_st = ns;
      s.n_gr = ng;
      s.abort = 0;
    }
  } else if (c == 0) {
    for (int b = tid - 32; b < p.B; b += kThreads - 32) {
      const int md = p.mode[b];
      bool bad = (md != 0 && md != 1) || (md == 1 && p.draft_probs == nullptr && p.n_draft[b] > 0);
      if (p.top_p != nullptr) {
        const float tp = __ldg(p.top_p + b);
        bad |= !(tp > 0.f && tp <= 1.f);
      }
      if (bad) atomicOr(p.status, SPADE_DEV_BAD_INDEX);
    }
  }
  block_sync();
  const int ns = s.n_st, ng = s.n_gr;
  const int ngroups = min(ns, nctas);
  const int gs = ns == 0 ? 1 : max(1, min(min(nctas / ngroups, kMaxGroup), (p.V + kMinShare - 1) / kMinShare));
  if (c < ngroups * gs) {
    const int g = c / gs, rank = c - g * gs;
    int lo, hi;
    share_of(p.V, gs, rank, &lo, &hi);
#pragma unroll 1
    for (int i = g; i < ns; i += ngroups) {
      const int b = s.st[i];
      const SeqInfo q = seq_info(p, b);
      decide_rows(p, s, b, q, rank == 0, warp, lane);
      const float top = seq_top_p(p, b);
      int upto = q.k;
      if (top < 1.f) {
        nucleus(p, s, b, q, top, g, rank, gs, lo, hi, tid, warp, lane);
        upto = min(q.k, s.nl);
      }
      const int a = first_reject(s, upto, tid);
      if (rank == 0 && tid == 0) p.accepted_len[b] = a;
      draw_token(p, s, b, q, a, g, rank, gs, lo, hi, p.kc != nullptr, tid, warp, lane);
      block_sync();
    }
  }
#pragma unroll 1
  for (int i = nctas - 1 - c; i < ng; i += nctas) {
    const int b = s.gr[i];
    const SeqInfo q = seq_info(p, b);
    if (!q.valid) {
      if (tid == 0) {
        p.accepted_len[b] = 0;
        p.next_token[b] = -1;
      }
      continue;
    }
    decide_rows(p, s, b, q, true, warp, lane);
    const int a = first_reject(s, q.k, tid);
    if (tid == 0) {
      p.accepted_len[b] = a;
      p.next_token[b] = s.arg[a];
    }
    if (p.kc != nullptr) commit_seq(p, b, q.k, a, tid);
    block_sync();
  }
}

}  // namespace accept
}  // namespace spade
