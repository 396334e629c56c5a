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
constexpr int kTBufBytes = kBlk * 32 * 4;           // one statistics warp's transpose buffer
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
  unsigned *bar;     // grid barrier words (kBarBytes)
  float4 *pstat;     // [R][NC]: slice max, slice sum-exp, slice argmax (bits), -
  float *ldraft;     // [R]: logit of the row's draft token
  float4 *gstat;     // [R]: merged row max, sum-exp, argmax (bits), accept bit
  float *logits;     // [R][ldl]: logits of the rows of sampled sequences (before temperature)
  unsigned long long *zpart;  // [2 attempts][B][kMaxGroup]: share masses of the sampled distribution (float-float)
  unsigned *nhist;   // [kNucRounds][kMaxGroup][R][kNucBins]: bin masses of the nucleus search (2^31 = all of p)
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
  int pool;  // bytes of RowsSmem::pool (nucleus search)
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

__device__ __forceinline__ unsigned long long ld_relaxed64(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(unsigned *p, unsigned v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed64(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Barrier words: the grid barrier's arrival count at word 0 and its generation
// in kReplicas copies, a 128-byte line each (CTA c polls copy c % kReplicas:
// 152 CTAs polling one line queue on it).
constexpr int kReplicas = 8;
constexpr int kGenWord = 32;
constexpr int kBarBytes = 2048;
static_assert(kGenWord * (kReplicas + 1) * 4 <= kBarBytes, "barrier words fit their region");
// Words that the CTAs of a group exchange (share masses, nucleus bins) are set to
// all ones before the statistics end; a reader polls the word itself until its
// writer has replaced it, so an exchange costs one store and one load through
// L2 (a barrier beside it: an atomic, a generation bump and a poll as well;
// 2.8 us against 1.3).
constexpr unsigned kUnset = 0xffffffffu;
constexpr unsigned long long kUnset64 = 0xffffffffffffffffull;
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
// Inclusive prefix sum over the warp's lanes.  (Rolled, one copy: the rows phase
// runs once after a long stream, and its cost is largely instruction fetch.)
static __device__ __noinline__ ff2 warp_scan_ff(ff2 v, int lane) {
#pragma unroll 1
  for (int o = 1; o < 32; o <<= 1) {
    const ff2 t{__shfl_up_sync(0xffffffffu, v.hi, o), __shfl_up_sync(0xffffffffu, v.lo, o)};
    if (lane >= o) v = ff_add(t, v);
  }
  return v;
}

// Device-wide barrier among the nctas co-resident CTAs (cooperative launch).  The
// last CTA to arrive resets the count and bumps the generation copies; the
// others poll theirs (relaxed loads with a short back-off, then an acquire
// fence) with a time limit.  Returns false if the wait expired.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, int nctas) {
  __shared__ int s_ok;
  block_sync();
  if (threadIdx.x == 0) {
    s_ok = 1;
    unsigned *gen_p = bar + kGenWord * (1 + blockIdx.x % kReplicas);
    // Read before arriving (the arrival's release orders this load first).
    const unsigned gen = ld_relaxed(gen_p);
    unsigned arrived;
    // The arrival releases this CTA's writes (ordered before it by bar.sync).
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(arrived) : "l"(bar) : "memory");
    if (arrived == static_cast<unsigned>(nctas) - 1) {
      st_relaxed(bar, 0u);
      // One release fence orders everything above before all the copies.
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      for (int r = 0; r < kReplicas; ++r)
        asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(bar + kGenWord * (1 + r)) : "memory");
    } else {
      const uint64_t t0 = globaltimer();
      while (ld_relaxed(gen_p) == gen) {
        if (globaltimer() - t0 > kWaitLimitNs) { s_ok = 0; break; }
        __nanosleep(20);
      }
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
    }
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

// Every sequence's rows and kind, in shared memory for the whole call.
struct SeqTable {
  int r0[kMaxB], k[kMaxB];
  unsigned valid[kMaxB / 32], stoch[kMaxB / 32];
  int st[kMaxB];  // sampled sequences, ascending
  int gr[kMaxB];  // greedy and invalid ones
  int n_st, n_gr;
  int rest;  // whether some row belongs to no valid sequence
  // This CTA among the groups that draw: groups, CTAs in each, its group and rank,
  // and its share [lo, hi) of the vocabulary.
  int ngroups, gs, g, rank, lo, hi;
};
__device__ __forceinline__ SeqInfo table_info(const SeqTable &t, int b) {
  const unsigned bit = 1u << (b % 32);
  return SeqInfo{t.r0[b], t.k[b], (t.valid[b / 32] & bit) != 0u, (t.stoch[b / 32] & bit) != 0u};
}
// Warp w of nw fills the words w, w + nw, ... (32 sequences each).
__device__ __forceinline__ void fill_table(const Call &p, SeqTable &t, int w, int nw, int lane, bool report) {
  for (int b0 = 32 * w; b0 < p.B; b0 += 32 * nw) {
    const int b = b0 + lane;
    SeqInfo q{0, 0, false, false};
    if (b < p.B) {
      q = seq_info(p, b);
      t.r0[b] = q.r0;
      t.k[b] = q.k;
      if (report) {
        const int md = p.mode[b];
        bool bad = !q.valid || (md != 0 && md != 1) || (md == 1 && p.draft_probs == nullptr && p.n_draft[b] > 0);
        if (p.top_p != nullptr) {
          const float tp = __ldg(p.top_p + b);
          bad |= !(tp > 0.f && tp <= 1.f);
        }
        if (bad) atomicOr(p.status, SPADE_DEV_BAD_INDEX);
      }
    }
    const unsigned mv = __ballot_sync(0xffffffffu, q.valid), ms = __ballot_sync(0xffffffffu, q.stoch);
    if (lane == 0) {
      t.valid[b0 / 32] = mv;
      t.stoch[b0 / 32] = ms;
    }
  }
}

// This CTA's share [lo, hi) of the vocabulary in a group of gs, shares a
// multiple of 4 entries (logits rows are read as float4).
__device__ __forceinline__ void share_of(int V, int gs, int rank, int *lo, int *hi) {
  const int per = ((V + gs - 1) / gs + 3) & ~3;
  *lo = min(V, rank * per);
  *hi = min(V, *lo + per);
}

// The lists of sampled and of other sequences and CTA c's place among nctas, by
// one warp, once the table is full.
__device__ __forceinline__ void fill_lists(const Call &p, SeqTable &t, int c, int nctas, int lane) {
  int ns = 0, ng = 0;
  unsigned invalid = 0u;
  for (int b0 = 0; b0 < p.B; b0 += 32) {
    const int b = b0 + lane;
    const unsigned in = p.B - b0 >= 32 ? 0xffffffffu : (1u << (p.B - b0)) - 1u;
    const unsigned ms = t.stoch[b0 / 32] & in, mg = ~t.stoch[b0 / 32] & in;
    invalid |= ~t.valid[b0 / 32] & in;
    const unsigned bit = 1u << lane, below = bit - 1u;
    if (ms & bit) t.st[ns + __popc(ms & below)] = b;
    if (mg & bit) t.gr[ng + __popc(mg & below)] = b;
    ns += __popc(ms);
    ng += __popc(mg);
  }
  if (lane == 0) {
    t.n_st = ns;
    t.n_gr = ng;
    // (valid sequences follow one another, so all of them cover the rows from the first's start on)
    t.rest = invalid != 0u || t.r0[0] != 0 || t.r0[p.B - 1] + t.k[p.B - 1] + 1 != p.R;
    t.ngroups = min(ns, nctas);
    t.gs = ns == 0 ? 1 : max(1, min(min(nctas / t.ngroups, kMaxGroup), (p.V + kMinShare - 1) / kMinShare));
    t.g = c / t.gs;
    t.rank = c - t.g * t.gs;
    share_of(p.V, t.gs, t.rank, &t.lo, &t.hi);
  }
}

// Per-row tables of the statistics epilogue, `nrows` entries each (a multiple of
// 16): row n = cu_q[b] + i is position i of sequence b; it holds draft i for i < k_b.
struct RowTables {
  int32_t *draft;   // draft token, -1: none
  float *it;        // 1 / T
  unsigned *keep;   // [nrows / 16]: bit n % 16 of word n / 16: the row's logits are kept for the draw
  float *u, *q;     // uniform and q(draft), or null: read by the rows phase itself
};
__host__ __device__ constexpr int row_table_bytes(int nrows, bool uq) {
  return nrows * (uq ? 16 : 8) + nrows / kBlk * 4;
}
__device__ __forceinline__ RowTables row_tables(uint8_t *mem, int nrows, bool uq) {
  RowTables t;
  t.draft = reinterpret_cast<int32_t *>(mem);
  t.it = reinterpret_cast<float *>(t.draft + nrows);
  t.u = uq ? t.it + nrows : nullptr;
  t.q = uq ? t.u + nrows : nullptr;
  t.keep = reinterpret_cast<unsigned *>((uq ? t.q : t.it) + nrows);
  return t;
}
// Filled by the epilogue warps (thread et of kN) while the first stages already
// stream.
template <int kN>
__device__ __forceinline__ void setup_rows(const Call &p, int nrows, SeqTable &seqs, const RowTables &t, int et) {
  for (int n = et; n < nrows; n += kN) { t.draft[n] = -1; t.it[n] = 1.f; }
  for (int w = et; w < nrows / kBlk; w += kN) t.keep[w] = 0u;
  fill_table(p, seqs, et / 32, (kN / 32), et % 32, true);
  named_bar(1, kN);
  // The rows' sequences (one warp per sequence), then one thread per row, so
  // that the loads of all rows are in flight together.
  for (int b = et / 32; b < p.B; b += (kN / 32)) {
    const SeqInfo q = table_info(seqs, b);
    if (!q.valid) continue;
    for (int i = et % 32; i <= q.k; i += 32) t.draft[q.r0 + i] = b;
  }
  if (et / 32 == kN / 32 - 1) fill_lists(p, seqs, blockIdx.x, p.NC, et % 32);  // (for the one-launch form's rows phase)
  named_bar(1, kN);
  for (int n = et; n < p.R; n += kN) {
    const int b = t.draft[n];
    if (b < 0) continue;
    const SeqInfo q = table_info(seqs, b);
    const int d = n - q.r0 < q.k ? p.draft_tokens[n - b] : -1;
    t.it[n] = inv_temp(p, b);
    t.draft[n] = d;
    if (q.stoch) atomicOr(&t.keep[n / kBlk], 1u << (n % kBlk));
    if (t.u) {
      t.u[n] = p.uniforms[n];
      t.q[n] = q.stoch && d >= 0 && d < p.V ? __ldg(&p.draft_probs[static_cast<size_t>(n - b) * p.V + d]) : 0.f;
    }
  }
  named_bar(1, kN);
}

// Sets the words that the rows phase's groups exchange to unset (thread i of n
// of the statistics launch; ordered before the rows phase by the grid barrier
// or the launch's end).
__device__ __forceinline__ void clear_exchange(const Call &p, int i, int n) {
  for (int e = i; e < 2 * p.B * kMaxGroup; e += n) p.zpart[e] = kUnset64;
  if (p.top_p != nullptr) {
    uint4 *h = reinterpret_cast<uint4 *>(p.nhist);
    const int words = kNucRounds * kMaxGroup * p.R * (kNucBins / 4);
    for (int e = i; e < words; e += n) h[e] = make_uint4(kUnset, kUnset, kUnset, kUnset);
  }
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

// Two fp32 operations in one instruction, each rounded as the scalar one.
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 f2_unpack(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Statistics of 16 verify rows (r0 ..) over one warp's 32 vocabulary entries
// (v0 + lane), `raw` the lane's accumulator columns.  A 16 x 32 shared-memory
// transpose (16-byte chunk j of row r at chunk j ^ (r % 8): the stores and the
// 16-byte loads are free of bank conflicts) gives lane (row = lane % 16,
// half = lane / 16) one row over 16 entries, reduced serially in pairs; the two
// halves meet by a shuffle each for the maximum and the sum.  The argmax search
// runs only when the block raises a row's running maximum.  Rows marked in
// `rows.keep` also store their logits, 128 contiguous bytes per row and warp.
__device__ __forceinline__ void stat_block(const Call &p, uint32_t (&raw)[kBlk], int r0, int v0, int v_hi,
                                           const RowTables &rows, float *T, int lane, BlkStat &st) {
  const int row = lane % kBlk, half = lane / kBlk, vb = half * kBlk;  // 16 entries from v0 + vb on
  const int n = r0 + row;
  const float it = rows.it[n];  // logits at the row's temperature, l / T
  const float rm = st.m[row];
  const int d = rows.draft[n] - (v0 + vb);
  const unsigned keep = rows.keep[r0 / kBlk];
  const bool whole = v0 + 32 <= v_hi;  // (warp-uniform)
  if (keep != 0u && v0 + lane < v_hi) {
    float *dst = p.logits + static_cast<size_t>(r0) * p.ldl + v0 + lane;
    if (keep == 0xffffu) {
#pragma unroll
      for (int r = 0; r < kBlk; ++r) dst[static_cast<size_t>(r) * p.ldl] = __uint_as_float(raw[r]);
    } else {
#pragma unroll
      for (int r = 0; r < kBlk; ++r)
        if ((keep >> r) & 1u) dst[static_cast<size_t>(r) * p.ldl] = __uint_as_float(raw[r]);
    }
  }
  if (!whole) {
#pragma unroll
    for (int r = 0; r < kBlk; ++r)
      if (v0 + lane >= v_hi) raw[r] = 0xff800000u;  // lanes past the slice: -infinity
  }
#pragma unroll
  for (int r = 0; r < kBlk; ++r) T[r * 32 + ((((lane >> 2) ^ (r & 7)) << 2) | (lane & 3))] = __uint_as_float(raw[r]);
  __syncwarp();
  uint64_t x[kBlk / 2];
  const uint64_t it2 = f2_pack(it, it);
#pragma unroll
  for (int j = 0; j < kBlk / 4; ++j) {
    const float4 v = *reinterpret_cast<const float4 *>(T + row * 32 + (((half * 4 + j) ^ (row & 7)) << 2));
    x[2 * j] = f2_mul(f2_pack(v.x, v.y), it2);
    x[2 * j + 1] = f2_mul(f2_pack(v.z, v.w), it2);
  }
  float m = -INFINITY, m1 = -INFINITY;
#pragma unroll
  for (int j = 0; j < kBlk / 2; ++j) {
    const float2 v = f2_unpack(x[j]);
    m = fmaxf(m, v.x);
    m1 = fmaxf(m1, v.y);
  }
  m = fmaxf(m, m1);
  m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, kBlk));
  const float M = fmaxf(rm, m);
  const float ref = M == -INFINITY ? 0.f : M;
  const uint64_t ref2 = f2_pack(-ref, -ref), log2e2 = f2_pack(kLog2e, kLog2e);
  uint64_t a2 = 0;
#pragma unroll
  for (int j = 0; j < kBlk / 2; ++j) {
    const float2 e = f2_unpack(f2_mul(f2_add(x[j], ref2), log2e2));
    a2 = f2_add(a2, f2_pack(ex2(e.x), ex2(e.y)));
  }
  const float2 a = f2_unpack(a2);
  float a0 = a.x + a.y;
  a0 += __shfl_xor_sync(0xffffffffu, a0, kBlk);
  const bool raised = m > rm;
  int idx = INT_MAX;
  if (__any_sync(0xffffffffu, raised)) {
#pragma unroll
    for (int j = kBlk / 2 - 1; j >= 0; --j) {
      const float2 v = f2_unpack(x[j]);
      if (v.y == m) idx = v0 + vb + 2 * j + 1;
      if (v.x == m) idx = v0 + vb + 2 * j;
    }
    idx = min(idx, __shfl_xor_sync(0xffffffffu, idx, kBlk));  // the lowest index of the maximum
  }
  if (lane < kBlk && M != -INFINITY) {
    st.s[row] = st.s[row] * ex2((rm - M) * kLog2e) + a0;
    if (raised) {
      st.m[row] = m;
      st.i[row] = idx;
    }
  }
  if (d >= 0 && d < kBlk && v0 + vb + d < v_hi)
    p.ldraft[n] = __fmul_rn(T[row * 32 + (((half * 4 + (d >> 2)) ^ (row & 7)) << 2) + (d & 3)], it);
  __syncwarp();
}

// The accumulator columns of a block (complete after tmem_wait_ld).
__device__ __forceinline__ void load_block(uint32_t taddr, uint32_t (&raw)[kBlk]) {
  tmem_ld8(taddr, raw);
  tmem_ld8(taddr + 8, raw + 8);
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
constexpr int kPiece = 8192;       // entries of a share that the draw takes at a time
constexpr int kMaxPieces = 80;     // 622592 entries, the largest vocabulary
struct RowsSmem {
  uint64_t bar[2];       // bulk copies of a piece, by buffer
  int first, nl, owner_piece, owner_warp, retry, abort;
  ff2 tgt, before;
  ff2 pm[kMaxPieces][kWarps];  // masses of the warps' parts of each piece of this CTA's share
  float m[kMaxR], z[kMaxR];           // rows of the sequence at hand: maximum, sum of exponentials
  float u[kMaxR], q[kMaxR], l[kMaxR]; // uniform, q(draft), draft logit
  int arg[kMaxR], d[kMaxR], ok[kMaxR];
  int tkey[kMaxR];       // nucleus key threshold (INT_MIN: all of p)
  union alignas(16) {
    float piece[2 * kPiece];  // a piece's logits (then its terms) and draft distribution: the first buffer
    float bins[kWarps][kNucSubs * kNucBins * 32];  // nucleus search
  };
  // Nucleus search only (one-launch path, at most 256 rows):
  int npre[kMaxRes];
  unsigned nab[kMaxRes];
  // Call::pool bytes: unsigned hist[rows][kNucBins], uint16_t cnt[items][32]
  // (list lengths per item and lane), float list[items][entries][32]; then, if it
  // is large enough, the draw's second buffer of a piece.
  alignas(16) uint8_t pool[16];
};
constexpr int kPieceBytes = 2 * kPiece * sizeof(float);
constexpr size_t kRowsBytesPlain = offsetof(RowsSmem, piece) + kPieceBytes;
constexpr size_t kRowsBytesDouble = offsetof(RowsSmem, pool) + kPieceBytes;
static_assert(offsetof(RowsSmem, piece) % 16 == 0, "bulk copies need 16-byte alignment");
constexpr int kPoolPerRow = kNucBins * 4 + 32 * 2;  // bins and list lengths of one searched row

// Bounded poll of an exchanged mass until its writer has set it.  After an
// expired wait of the CTA every later poll gives up at once.
__device__ __forceinline__ ff2 poll_mass(const Call &p, RowsSmem &s, const unsigned long long *a) {
  unsigned long long v = ld_relaxed64(a);
  if (v == kUnset64) {
    const uint64_t t0 = globaltimer();
    while ((v = ld_relaxed64(a)) == kUnset64) {
      if (*const_cast<volatile int *>(&s.abort)) return ff2{0.f, 0.f};
      if (globaltimer() - t0 > kWaitLimitNs) {
        *const_cast<volatile int *>(&s.abort) = 1;
        atomicOr(p.status, SPADE_DEV_TIMEOUT);
        return ff2{0.f, 0.f};
      }
    }
  }
  return ff2{__uint_as_float(static_cast<unsigned>(v)), __uint_as_float(static_cast<unsigned>(v >> 32))};
}
__device__ __forceinline__ void post_mass(unsigned long long *a, ff2 z) {
  // (a NaN mass must not read as unset: lo is then zero)
  const unsigned lo = z.lo == z.lo ? __float_as_uint(z.lo) : 0u;
  st_relaxed64(a, static_cast<unsigned long long>(lo) << 32 | __float_as_uint(z.hi));
}

// A row's merged statistics over the NC slice partials (in `part`, lane by lane):
// the maximum first, then its lowest index and the rescaled sum.  lane 0's values count.
constexpr int kPartLoads = kMaxNC / 32;
__device__ __forceinline__ void load_parts(const Call &p, int n, int lane, float4 (&part)[kPartLoads]) {
#pragma unroll
  for (int j = 0; j < kPartLoads; ++j) {
    const int cc = j * 32 + lane;
    part[j] = cc < p.NC ? __ldcg(&p.pstat[static_cast<size_t>(n) * p.NC + cc])
                        : make_float4(-INFINITY, 0.f, __int_as_float(INT_MAX), 0.f);
  }
}
__device__ __forceinline__ void merge_parts(const float4 (&part)[kPartLoads], float &m, float &z, int &idx) {
  m = -INFINITY;
#pragma unroll
  for (int j = 0; j < kPartLoads; ++j) m = fmaxf(m, part[j].x);
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  z = 0.f;
  idx = INT_MAX;
  if (m != -INFINITY) {
#pragma unroll
    for (int j = 0; j < kPartLoads; ++j) {
      z += part[j].y * ex2((part[j].x - m) * kLog2e);
      if (part[j].x == m) idx = min(idx, __float_as_int(part[j].z));
    }
  }
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    z += __shfl_xor_sync(0xffffffffu, z, o);
    idx = min(idx, __shfl_xor_sync(0xffffffffu, idx, o));
  }
}

// Statistics of the rows that belong to no valid sequence (past cu_q[B], or of a
// sequence that was reported), with accept bit 0; one warp per row.
__device__ __forceinline__ void rest_rows(const Call &p, const SeqTable &seqs, int c, int nctas, int warp, int lane) {
#pragma unroll 1
  for (int n = c * kWarps + warp; n < p.R; n += nctas * kWarps) {
    bool taken = false;
    for (int b = lane; b < p.B; b += 32) {
      const SeqInfo q = table_info(seqs, b);
      taken |= q.valid && n >= q.r0 && n <= q.r0 + q.k;
    }
    if (__any_sync(0xffffffffu, taken)) continue;
    float4 part[kPartLoads];
    load_parts(p, n, lane, part);
    float m, z;
    int idx;
    merge_parts(part, m, z, idx);
    if (lane == 0) __stcg(&p.gstat[n], make_float4(m, z, __int_as_float(idx), __int_as_float(0)));
  }
}

// Merged statistics and accept bits of the rows of sequence b, one warp per
// row over the NC slice partials.  Greedy: the draft is the argmax (lowest
// index on ties); stochastic: u < p(d) / q(d) (Sec. III-C).
__device__ __forceinline__ void decide_rows(const Call &p, RowsSmem &s, const RowTables &rows, int b, const SeqInfo &q,
                                            bool writer, int warp, int lane) {
#pragma unroll 1
  for (int i = warp; i <= q.k; i += kWarps) {
    const int n = q.r0 + i;
    float4 part[kPartLoads];
    load_parts(p, n, lane, part);
    int d = -1;
    float u = 0.f, qd = 0.f, ld = 0.f;
    if (i < q.k) {
      if (rows.u) {  // read while the vocabulary streamed
        ld = __ldcg(&p.ldraft[n]);
        d = rows.draft[n];
        u = rows.u[n];
        qd = rows.q[n];
      } else {
        d = p.draft_tokens[n - b];
        ld = __ldcg(&p.ldraft[n]);
        u = p.uniforms[n];
        if (q.stoch && d >= 0 && d < p.V) qd = __ldg(&p.draft_probs[static_cast<size_t>(n - b) * p.V + d]);
      }
    }
    float m, z;
    int idx;
    merge_parts(part, m, z, idx);
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

// Adds four values of a row to a lane's bins.  `v` holds scaled logits; a value
// counts when `in` says so and its key has the prefix bits.
struct BinRound {
  float nb65, mlog;
  int sh, pre_bits;
};
__device__ __forceinline__ void bin4(const BinRound &t, float *bins, const float (&l)[4], const bool (&in)[4]) {
  float ex[4];
  int a[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int kbits = nuc_key_bits(l[c], t.nb65);
    const bool hit = in[c] && (kbits >> (t.sh + kNucBinBits)) == t.pre_bits;
    ex[c] = hit ? ex2(__fmaf_rn(l[c], kLog2e, t.mlog)) : 0.f;
    a[c] = ((c % kNucSubs) * kNucBins + ((kbits >> t.sh) & (kNucBins - 1))) * 32;
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

// Top-p: the nucleus of the rows of sequence b that can decide anything (see
// nuc_key), its group together.  A draft row whose u is past p(d) / (top_p q(d))
// is rejected whatever its nucleus (the nucleus holds at least top_p of p), so
// the rows after the first such row are not searched.  Per round every CTA bins
// its share of each row -- lane-private fp32 bins in kNucSubs copies (lane i's
// words all in bank i: no conflicts, no shared-memory atomics per value), summed
// in a fixed order and added to the row's bins in fixed point (2^31 = all of p:
// integer sums, the same in any order) -- posts them, and sums every CTA's bins
// itself as they arrive.
// The first round bins every value and is bound by its ~18 instructions each.
// The second keeps the values of the chosen bin (one unit of log-probability
// wide: a few percent of a row) in lane-private lists, and it and the later
// rounds bin only those; an item whose list overflows reads its values again.
__device__ __forceinline__ void nucleus(const Call &p, RowsSmem &s, int b, const SeqInfo &q, float top, int rank,
                                        int gs, int lo, int hi, int tid, int warp, int lane) {
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
  const int items = nl * parts;
  const int per = ((hi - lo + parts - 1) / parts + 127) & ~127;
  unsigned(*hist)[kNucBins] = reinterpret_cast<unsigned(*)[kNucBins]>(s.pool);
  uint16_t(*cnt)[32] = reinterpret_cast<uint16_t(*)[32]>(s.pool + nl * kNucBins * 4);
  float *lists = reinterpret_cast<float *>(s.pool + nl * kNucBins * 4 + items * 32 * 2);
  // List entries per lane and item.
  const int cap = min(4096, (p.pool - nl * kNucBins * 4 - items * 32 * 2) / (32 * 4 * items));
  float *bins = s.bins[warp] + lane;
#pragma unroll 1
  for (int r = 0; r < kNucRounds; ++r) {
    const int sh = kNucKeyBits - kNucBinBits * (r + 1);  // this round's bin: key bits [sh, sh + 5)
    for (int e = tid; e < nl * kNucBins; e += kThreads) hist[e / kNucBins][e % kNucBins] = 0u;
    block_sync();
#pragma unroll 1
    for (int item = warp; item < items; item += kWarps) {
      const int i = item / parts, part = item - i * parts;
      const int pre = s.npre[i];
      if (pre < 0) continue;
      const float M = s.m[i];
      BinRound t;
      t.nb65 = -kNucScale * __fsub_rn(M, kNucSpan);
      t.mlog = -M * kLog2e;
      t.sh = sh;
      t.pre_bits = pre + (kNucKeyBias >> (sh + kNucBinBits));  // the range's key prefix, as bits
      const float *lg = p.logits + static_cast<size_t>(q.r0 + i) * p.ldl;
      const int plo = lo + part * per, phi = min(hi, plo + per);
      float *list = lists + item * cap * 32 + lane;  // entry j of this lane: list[32 j]
      int n = r == 0 ? cap + 1 : (r == 1 ? 0 : cnt[item][lane]);
#pragma unroll 8
      for (int k = 0; k < kNucSubs * kNucBins; ++k) bins[k * 32] = 0.f;
      if (r == 1) {
        // Values with the first round's prefix, kept (past cap only counted).
#pragma unroll 1
        for (int e0 = plo + 4 * lane; e0 < phi; e0 += 4 * 128) {
          float4 v4[4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            v4[j] = e0 + 128 * j < phi ? __ldcg(reinterpret_cast<const float4 *>(lg + e0 + 128 * j))
                                       : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float x[4] = {v4[j].x, v4[j].y, v4[j].z, v4[j].w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              const float l = __fmul_rn(x[c], IT);
              const bool in = e0 + 128 * j + c < phi &&
                              (nuc_key_bits(l, t.nb65) >> (sh + kNucBinBits)) == t.pre_bits;
              if (in) {
                if (n < cap) list[32 * n] = l;
                ++n;
              }
            }
          }
        }
        cnt[item][lane] = static_cast<uint16_t>(min(n, cap + 1));
      }
      if (__any_sync(0xffffffffu, n > cap)) {
#pragma unroll 1
        for (int e0 = plo + 4 * lane; e0 < phi; e0 += 4 * 128) {
          float4 v4[4];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            v4[j] = e0 + 128 * j < phi ? __ldcg(reinterpret_cast<const float4 *>(lg + e0 + 128 * j))
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int e = e0 + 128 * j;
            const float l[4] = {__fmul_rn(v4[j].x, IT), __fmul_rn(v4[j].y, IT), __fmul_rn(v4[j].z, IT),
                                __fmul_rn(v4[j].w, IT)};
            const bool in[4] = {e < phi, e + 1 < phi, e + 2 < phi, e + 3 < phi};
            bin4(t, bins, l, in);
          }
        }
      } else {
#pragma unroll 1
        for (int j = 0; j < n; j += 4) {
          float l[4];
          bool in[4];
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            in[c] = j + c < n;
            l[c] = in[c] ? list[32 * (j + c)] : 0.f;
          }
          bin4(t, bins, l, in);
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
      if (fixed != 0u) atomicAdd(&hist[i][lane], fixed);
      __syncwarp();
    }
    block_sync();
    unsigned *round = p.nhist + (static_cast<size_t>(r * kMaxGroup) * p.R + q.r0) * kNucBins;
    const size_t stride = static_cast<size_t>(p.R) * kNucBins;  // words between the CTAs' bins
    if (gs > 1)
      for (int e = tid; e < nl * kNucBins; e += kThreads)
        st_relaxed(round + rank * stride + e, hist[e / kNucBins][e % kNucBins]);
    // C_k = mass of keys at or above bin k plus the mass above the range: keep
    // the highest bin with C_k >= top_p.  Sums stay below 2^33.
#pragma unroll 1
    for (int i = warp; i < nl; i += kWarps) {
      unsigned long long own = hist[i][lane];
      if (gs > 1) {
        const unsigned *src = round + i * kNucBins + lane;
        unsigned v[kMaxGroup];  // every CTA's bins in flight at once
#pragma unroll
        for (int c = 0; c < kMaxGroup; ++c) v[c] = c < gs && c != rank ? ld_relaxed(src + c * stride) : 0u;
        // The late ones again, all in flight at once (one after the other, a round
        // spent 5 us here with 19 CTAs).
        uint64_t t0 = 0;
#pragma unroll 1
        for (;;) {
          bool late = false;
#pragma unroll
          for (int c = 0; c < kMaxGroup; ++c) late |= v[c] == kUnset;
          if (!__any_sync(0xffffffffu, late)) break;
          const uint64_t now = globaltimer();
          if (t0 == 0) t0 = now;
          const bool expired = now - t0 > kWaitLimitNs;
          if (__any_sync(0xffffffffu, expired || *const_cast<volatile int *>(&s.abort))) {
            *const_cast<volatile int *>(&s.abort) = 1;
            atomicOr(p.status, SPADE_DEV_TIMEOUT);
            break;
          }
#pragma unroll
          for (int c = 0; c < kMaxGroup; ++c)
            if (v[c] == kUnset) v[c] = ld_relaxed(src + c * stride);
        }
        __syncwarp();
#pragma unroll
        for (int c = 0; c < kMaxGroup; ++c) own += v[c] == kUnset ? 0u : v[c];
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
};
// Entries of a lane's block of a piece of `len` entries: the ten warps take
// contiguous parts, their lanes contiguous blocks of an odd length (lanes then
// read distinct banks).
__device__ __forceinline__ int lane_block(int len) { return ((len + kThreads - 1) / kThreads) | 1; }

__device__ __forceinline__ float *piece_buf(RowsSmem &s, int buf) {
  return buf == 0 ? s.piece : reinterpret_cast<float *>(s.pool);
}
// Issues the bulk copies of entries [e0, e0 + len) of the logits row (and of q) into
// a buffer that no thread uses (warp kCopyWarp, after a barrier; a whole warp, as
// the copies' operands live in uniform registers).
constexpr int kCopyWarp = 2;  // (on a scheduler with two of the ten warps)
__device__ __forceinline__ void piece_copy(const Call &p, RowsSmem &s, const Dist &t, int e0, int len, int buf) {
  float *sl = piece_buf(s, buf);
  const bool leader = elect_one(), bulk_q = t.q != nullptr && p.qvec;
  const uint32_t bytes = static_cast<uint32_t>(uniform((len + 3) & ~3)) * 4u;
  const float *lsrc = uniform(t.lg + e0), *qsrc = uniform(t.q + e0);
  if (leader) {
    fence_proxy_async();  // earlier generic accesses, and the logits' stores, come first
    mbar_arrive_expect_tx(&s.bar[buf], bulk_q ? 2 * bytes : bytes);
    bulk_load(sl, lsrc, bytes, &s.bar[buf]);
    if (bulk_q) bulk_load(sl + kPiece, qsrc, bytes, &s.bar[buf]);
  }
  __syncwarp();
}
// Waits for a piece, replaces its logits by the terms of the distribution and
// returns the inclusive prefix of this lane's block sum over the warp.  (q comes by
// plain loads when its rows are not 16-byte aligned.)
// The terms are fp32; sums are compensated (the terms are >= 0, so ordering the
// two addends by size makes the error term exact).
__device__ __forceinline__ ff2 piece_terms(const Call &p, RowsSmem &s, const Dist &t, int e0, int len, int buf,
                                           uint32_t parity, int tid, int warp, int lane) {
  float *sl = piece_buf(s, buf), *sq = sl + kPiece;
  if (t.q != nullptr && !p.qvec) {
#pragma unroll 4
    for (int e = tid; e < len; e += kThreads) sq[e] = __ldg(t.q + e0 + e);
  }
  // (the copies read valid memory: this wait does not give up on an earlier
  // expired wait, so that no copy is left in flight at exit)
  if (!mbar_wait_unabortable(&s.bar[buf], parity)) {
    atomicOr(p.status, SPADE_DEV_TIMEOUT);
    s.abort = 1;
  }
  block_sync();
  const int bs = lane_block(len);
  const int b0 = (warp * 32 + lane) * bs, b1 = min(len, b0 + bs);
  float sh = 0.f, lo = 0.f;
  // Four entries' loads come before any of their stores (entry by entry, each load
  // waits for the store before it); bound by its ~17 instructions an entry.
  const float nM = -t.M;
#pragma unroll 1
  for (int e = b0; e < b1; e += 4) {
    float x[4], qx[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool in = e + j < b1;
      x[j] = in ? sl[e + j] : -INFINITY;
      qx[j] = in && t.q != nullptr ? sq[e + j] : 0.f;
    }
    float pv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[j] = __fmul_rn(x[j], t.IT);
      pv[j] = ex2((x[j] + nM) * kLog2e) * t.invS;
    }
    if (t.tkey != INT_MIN) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (nuc_key(x[j], t.base) < t.tkey) pv[j] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float v = t.q != nullptr ? fmaxf(0.f, pv[j] - qx[j]) : pv[j];
      if (e + j < b1) {
        sl[e + j] = v;
        const float sm = sh + v;
        lo += (fmaxf(sh, v) - sm) + fminf(sh, v);
        sh = sm;
      }
    }
  }
  return warp_scan_ff(ff_norm(sh, lo), lane);
}

// The draw of sequence b by its group: next_token[b] is the first entry whose
// cumulative mass exceeds u Z.  Terms are fp32, every sum float-float, so the
// cumulative masses that place u Z are as exact as the terms allow.  The shares'
// masses meet in the workspace, every CTA finds the owner of u Z from the same
// masses, and the owner walks down: piece, warp, lane block, entry.  A residual
// with no mass is retried on p (every CTA sees the same total, so all retry
// together).  Bound by the latency of its few dependent steps, and by fetching
// its code: loops are rolled.
// A share of more than one piece has the next piece's copies in flight under this
// one's sums where shared memory holds two (389 rows, 32 of 64 sequences sampled,
// shares of 38016 entries: the second launch 30 -> 26 us with that and terms taken four at a time).
// `commit`: the group's first CTA updates the cache while the masses travel.
// `parity`: phases of the buffers' mbarriers (bit: buffer), flipped by every piece.
__device__ __forceinline__ void draw_token(const Call &p, RowsSmem &s, int b, const SeqInfo &q, int a, int rank, int gs,
                                           int lo, int hi, bool commit, uint32_t &parity, int tid, int warp,
                                           int lane) {
  const int n = q.r0 + a;
  Dist t;
  t.lg = p.logits + static_cast<size_t>(n) * p.ldl;
  t.q = a < q.k ? p.draft_probs + static_cast<size_t>(n - b) * p.V : nullptr;
  t.M = s.m[a];
  t.invS = 1.f / s.z[a];
  t.IT = inv_temp(p, b);
  t.base = __fsub_rn(t.M, kNucSpan);
  t.tkey = s.tkey[a];
  const float u = p.uniforms[q.r0 + q.k];
  const int npiece = (hi - lo + kPiece - 1) / kPiece;
  const int nbuf = p.pool >= kPieceBytes ? 2 : 1;
  auto copy = [&](int j) {
    if (warp == kCopyWarp && j < npiece) piece_copy(p, s, t, lo + j * kPiece, min(kPiece, hi - lo - j * kPiece), j % nbuf);
  };
  ff2 incl;
  int i = 0, attempt = 0;
  bool again = false;  // the owner takes the piece that holds the target once more
  for (int j = 0; j < nbuf; ++j) copy(j);
#pragma unroll 1
  for (;;) {  // (one copy of the piece's code)
    const int buf = i % nbuf;
    incl = piece_terms(p, s, t, lo + i * kPiece, min(kPiece, hi - lo - i * kPiece), buf, (parity >> buf) & 1u, tid, warp,
                       lane);
    parity ^= 1u << buf;
    if (again) break;
    if (lane == 31) s.pm[i][warp] = incl;
    block_sync();
    copy(i + nbuf);
    if (++i < npiece) continue;
    ff2 share{0.f, 0.f};
    unsigned long long *zp = p.zpart + (static_cast<size_t>(attempt) * p.B + b) * kMaxGroup;
    if (warp == 0) {
      // This share's mass: lane w sums the pieces of warp w's parts, in order.
      ff2 z{0.f, 0.f};
      for (int j = 0; j < npiece && lane < kWarps; ++j) z = ff_add(z, s.pm[j][lane]);
      share = ff_shfl(warp_scan_ff(z, lane), 31);
      if (lane == 0 && gs > 1) post_mass(&zp[rank], share);
    }
    if (attempt == 0 && commit && rank == 0) commit_seq(p, b, q.k, a, tid);
    if (warp == 0) {
      const ff2 mine = gs == 1 && lane == 0 ? share : (gs > 1 && lane < gs ? poll_mass(p, s, &zp[lane]) : ff2{0.f, 0.f});
      __syncwarp();
      const ff2 reach = warp_scan_ff(mine, lane);
      const ff2 tot = ff_shfl(reach, 31);
      const bool ok = tot.hi > 0.f && isfinite(tot.hi);
      const ff2 target = ff_mul_f(tot, u);
      const unsigned hit = __ballot_sync(0xffffffffu, ok && mine.hi > 0.f && ff_gt(reach, target));
      const unsigned pos = __ballot_sync(0xffffffffu, ok && mine.hi > 0.f);
      // Rounding past the total clamps to the last share with mass.
      const int own = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : -1);
      const ff2 before = ff_shfl(ff_sub(reach, mine), own < 0 ? 0 : own);
      int own_piece = -1, own_warp = 0;
      if (own == rank) {
        // The piece, then the warp part, in vocabulary order; rounding past the
        // share's mass clamps to the last part with mass.
        ff2 left = hit ? ff_sub(target, before) : ff2{INFINITY, 0.f};
        ff2 run{0.f, 0.f}, left_at = left;
        bool over = false;
#pragma unroll 1
        for (int j = 0; j < npiece && !over; ++j) {
          const ff2 wm = lane < kWarps ? s.pm[j][lane] : ff2{0.f, 0.f};
          const ff2 wr = ff_add(run, warp_scan_ff(wm, lane));
          const unsigned wh = __ballot_sync(0xffffffffu, wm.hi > 0.f && ff_gt(wr, left));
          const unsigned wp = __ballot_sync(0xffffffffu, wm.hi > 0.f);
          const int w = wh ? __ffs(wh) - 1 : (wp ? 31 - __clz(wp) : -1);
          over = wh != 0u;
          if (w >= 0) {
            own_piece = j;
            own_warp = w;
            left_at = over ? ff_sub(left, ff_shfl(ff_sub(wr, wm), w)) : ff2{INFINITY, 0.f};
          }
          run = ff_shfl(wr, 31);
        }
        if (lane == 0) s.tgt = left_at;  // target left inside the warp's part
      }
      if (lane == 0) {
        s.retry = !ok;
        s.owner_piece = own_piece;
        s.owner_warp = own_warp;
        if (!ok && attempt == 1 && rank == 0) p.next_token[b] = -1;  // p has no mass either
        if (ok && attempt == 1 && rank == 0) atomicOr(p.status, SPADE_DEV_FALLBACK);
      }
    }
    block_sync();
    if (s.retry) {  // the residual has no mass: sample p
      if (attempt == 1) return;
      attempt = 1;
      t.q = nullptr;
      i = 0;
      for (int j = 0; j < nbuf; ++j) copy(j);
      continue;
    }
    if (s.owner_piece < 0) return;
    if (s.owner_piece == npiece - 1) break;
    i = s.owner_piece;
    copy(i);
    again = true;
  }
  const int e0 = lo + s.owner_piece * kPiece, len = min(kPiece, hi - e0);
  const float *terms = piece_buf(s, s.owner_piece % nbuf);
  if (warp != s.owner_warp) return;
  __syncwarp();  // a piece taken again: its terms were stored lane by lane, the walk below reads another lane's
  // The lane block, then the entry.
  const ff2 left = s.tgt;
  const ff2 prev{__shfl_up_sync(0xffffffffu, incl.hi, 1), __shfl_up_sync(0xffffffffu, incl.lo, 1)};
  const bool some = lane == 0 ? incl.hi > 0.f : ff_gt(incl, prev);
  const unsigned hit = __ballot_sync(0xffffffffu, some && ff_gt(incl, left));
  const unsigned pos = __ballot_sync(0xffffffffu, some);
  const int blk = hit ? __ffs(hit) - 1 : (pos ? 31 - __clz(pos) : 0);
  const ff2 before = blk == 0 ? ff2{0.f, 0.f} : ff_shfl(incl, blk - 1);
  const int bs = lane_block(len), b0 = (warp * 32 + blk) * bs, b1 = min(len, b0 + bs);
  ff2 run = before;
  int token = -1;
  bool over = false;
#pragma unroll 1
  for (int c = b0; c < b1 && !over; c += 32) {
    const int e = c + lane;
    const float x = e < b1 ? terms[e] : 0.f;
    const ff2 reach = ff_add(run, warp_scan_ff(ff2{x, 0.f}, lane));
    const unsigned xh = __ballot_sync(0xffffffffu, hit != 0u && x > 0.f && ff_gt(reach, left));
    const unsigned xp = __ballot_sync(0xffffffffu, x > 0.f);
    over = xh != 0u;
    if (xp) token = e0 + c + (over ? __ffs(xh) - 1 : 31 - __clz(xp));  // else the last entry with mass
    run = ff_shfl(reach, 31);
  }
  if (lane == 0) p.next_token[b] = token >= 0 ? token : e0 + b0;
}

// After the statistics of every slice (a grid barrier, or the previous launch's
// end): decisions, outputs, commit and the draws.  Sampled sequences are dealt
// to groups of CTAs from the front of the grid, greedy ones to single CTAs
// from its end; no group waits for another.  The CTAs of a group wait for one
// another's words (every CTA is resident: cooperative launches, or one cluster).
__device__ __forceinline__ void rows_phase(const Call &p, RowsSmem &s, const SeqTable &seqs, const RowTables &rows, int c,
                                           int nctas) {
  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  // (every sequence's decisions meet at barriers before the first copy or poll)
  if (tid == 0) {
    s.abort = 0;
    mbar_init(&s.bar[0], 1);
    mbar_init(&s.bar[1], 1);
    fence_mbar_init();
  }
  const int ns = seqs.n_st, ng = seqs.n_gr;
  const int ngroups = seqs.ngroups, gs = seqs.gs;
  if (seqs.g < ngroups) {
    const int g = seqs.g, rank = seqs.rank, lo = seqs.lo, hi = seqs.hi;
    uint32_t parity = 0;
#pragma unroll 1
    for (int i = g; i < ns; i += ngroups) {
      const int b = seqs.st[i];
      const SeqInfo q = table_info(seqs, b);
      decide_rows(p, s, rows, b, q, rank == 0, warp, lane);
      const float top = seq_top_p(p, b);
      int upto = q.k;
      if (top < 1.f) {
        nucleus(p, s, b, q, top, rank, gs, lo, hi, tid, warp, lane);
        upto = min(q.k, s.nl);
      }
      const int a = first_reject(s, upto, tid);
      if (rank == 0 && tid == 0) p.accepted_len[b] = a;
      draw_token(p, s, b, q, a, rank, gs, lo, hi, p.kc != nullptr, parity, tid, warp, lane);
      block_sync();
    }
  }
#pragma unroll 1
  for (int i = nctas - 1 - c; i < ng; i += nctas) {
    const int b = seqs.gr[i];
    const SeqInfo q = table_info(seqs, b);
    if (!q.valid) {
      if (tid == 0) {
        p.accepted_len[b] = 0;
        p.next_token[b] = -1;
      }
      continue;
    }
    decide_rows(p, s, rows, b, q, true, warp, lane);
    const int a = first_reject(s, q.k, tid);
    if (tid == 0) {
      p.accepted_len[b] = a;
      p.next_token[b] = s.arg[a];
    }
    if (p.kc != nullptr) commit_seq(p, b, q.k, a, tid);
    block_sync();
  }
  if (seqs.rest) rest_rows(p, seqs, c, nctas, warp, lane);
}

}  // namespace accept
}  // namespace spade
