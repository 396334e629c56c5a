// verify_accept.cu -- LM head o = g(x_L) and softmax (Sec. III-A) fused with the
// accept test alpha(x) = min(1, p(x)/q(x)) and the residual sampling from
// p'(x) = norm(max(0, p(x) - q(x))) (Sec. III-C), i.e. the verify / accept /
// correct steps of Algorithm 1 for every sequence of the batch.  This file holds
// the one-launch form (see one_launch()) and the entry points; larger
// calls take lm_head_pairs.cu and accept_rows.cu.
//
// Design (GB300):
//  * The contraction logits[r, x] = hidden[r, :] . W[x, :] runs on the 5th-gen
//    tensor cores (tcgen05.mma kind::f16, bf16 in, fp32 accumulators in TMEM).
//    The vocabulary is the M side of the MMA (128 vocab rows per tile) and the
//    R verify rows are the N side, so W -- the only large operand -- streams
//    from HBM exactly once while the few hidden rows are re-read from L2.
//  * W and hidden arrive by TMA in 32 KB boxes: a 3-D view of the row-major
//    matrix fetches 128 rows x 2 k-chunks at once and lands them as two
//    canonical 128B-swizzled K-major tiles (a 2-D view covers a ragged tail).
//  * One CTA per SM (cooperative launch) owns a contiguous vocabulary slice and
//    takes its tiles in rounds of as many as half of the tensor memory holds:
//    a round's tiles share each load of the hidden rows, and the two halves
//    alternate, so the statistics of a round run under the next one's stream.
//  * Warp roles: warp 0 issues TMA loads, warp 1 owns TMEM and issues the
//    MMAs from a single thread, warps 2-9 (two per lane quarter) read the
//    accumulators back (tcgen05.ld), reduce per-row max / sum-exp / argmax across
//    the vocabulary and store the logits of the rows a sampled sequence may
//    draw from (37 MB at 72 rows x 128256 entries: most of it stays in L2, and
//    the phases after the stream read it in row order, by any CTA, where
//    tensor memory holds each CTA to its own slice and lane quarters).
//  * After one bounded device-wide barrier (a cluster barrier for grids of up to
//    eight CTAs) the rows phase (accept_common.cuh) takes the decisions, commits
//    and draws: groups of CTAs per sequence, exchanging polled words.
#include <atomic>

#include "accept_common.cuh"
#include "accept_launch.h"

namespace spade {
namespace accept {

constexpr int kMaxRounds = 32;
constexpr int kMaxTilesPerCta = 32;
constexpr int kHalfCols = kTmemCols / 2;  // accumulator columns of one round

struct Params {
  Call c;
  int T, Ncols;
  int KC;            // k-chunks of 64 (the last may be partial)
  int KCF;           // full k-chunks (H / 64)
  int KG;            // k-chunks per pipeline stage
  int NS;            // pipeline stages per round = ceil(KC / KG)
  int nrounds;
  int round_tiles[kMaxRounds];
  int HS, WS;        // hidden / W ring slots
  int BRS;           // box rows of the map used for a slice's last, partial tile
  uint32_t idesc;
};

struct Smem {
  int w_slot, h_slot;
  int off_h, off_bar, off_misc, off_seq, off_rows, off_stat, off_tbuf, total;
};

__host__ __device__ inline Smem smem_layout(const Params &p) {
  Smem s;
  s.w_slot = p.KG * kWChunkBytes;
  s.h_slot = p.KG * p.Ncols * 128;
  s.off_h = p.WS * s.w_slot;
  s.off_bar = s.off_h + p.HS * s.h_slot;  // the rings end here; the rows phase reuses them
  s.off_misc = (s.off_bar + (2 * p.WS + 2 * p.HS + 4) * 8 + 127) & ~127;
  s.off_seq = s.off_misc + 64;
  s.off_rows = s.off_seq + static_cast<int>(sizeof(SeqTable));
  s.off_stat = s.off_rows + row_table_bytes(p.Ncols, true);
  s.off_tbuf = (s.off_stat + kEpiWarps * (p.Ncols / kBlk) * static_cast<int>(sizeof(BlkStat)) + 127) & ~127;
  s.total = s.off_tbuf + kEpiWarps * kTBufBytes + 1024;
  return s;
}

// kCluster: the grid is one cluster (see launch()).
template <bool kCluster>
__global__ void __launch_bounds__(kThreads, 1) verify_accept_kernel(
    const __grid_constant__ Params p, const __grid_constant__ CUtensorMap tm_w3,
    const __grid_constant__ CUtensorMap tm_w2, const __grid_constant__ CUtensorMap tm_w2s,
    const __grid_constant__ CUtensorMap tm_w3s, const __grid_constant__ CUtensorMap tm_h3,
    const __grid_constant__ CUtensorMap tm_h2) {
  extern __shared__ uint8_t smem_raw[];
  // 1024-byte aligned base, derived by pointer arithmetic so that the compiler
  // keeps the shared state space (plain ld/st.shared, not generic accesses).
  uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const Smem L = smem_layout(p);
  uint8_t *w_ring = smem;
  uint8_t *h_ring = smem + L.off_h;
  uint64_t *w_full = reinterpret_cast<uint64_t *>(smem + L.off_bar);
  uint64_t *w_empty = w_full + p.WS;
  uint64_t *h_full = w_empty + p.WS;
  uint64_t *h_empty = h_full + p.HS;
  uint64_t *acc_full = h_empty + p.HS;  // [2]: one per tensor-memory half
  uint64_t *acc_empty = acc_full + 2;   // [2]
  volatile int *s_abort = reinterpret_cast<volatile int *>(smem + L.off_misc);
  uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L.off_misc + 8);
  SeqTable &seqs = *reinterpret_cast<SeqTable *>(smem + L.off_seq);
  const RowTables rows = row_tables(smem + L.off_rows, p.Ncols, true);

  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int c = blockIdx.x;
  // This CTA's vocabulary slice [v_lo, v_hi): equal row counts (within one),
  // cut into 128-row tiles; the last tile may be partial.
  const int v_lo = static_cast<int>(static_cast<int64_t>(c) * p.c.V / p.c.NC);
  const int v_hi = static_cast<int>(static_cast<int64_t>(c + 1) * p.c.V / p.c.NC);
  const int ntiles = (v_hi - v_lo + kTileV - 1) / kTileV;
  const bool short_last = (v_hi - v_lo) - (ntiles - 1) * kTileV <= p.BRS && p.BRS < kTileV;

  // ---- set-up that reads no input ------------------------------------------
  if (tid == 0) {
    *s_abort = 0;
    for (int s = 0; s < p.WS; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], 1); }
    for (int s = 0; s < p.HS; ++s) { mbar_init(&h_full[s], 1); mbar_init(&h_empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], kEpiWarps); }
    fence_mbar_init();
    tma_prefetch_desc(&tm_w3);
    tma_prefetch_desc(&tm_w3s);
    tma_prefetch_desc(&tm_h3);
  }
  if (warp == 1) {
    tmem_alloc(s_tmem, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  block_sync();
  tc_fence_after();
  // Inputs (and the workspace's contents) of earlier kernels in the stream are
  // visible from here on; the next kernel may be scheduled as this one's CTAs exit.
  griddep_wait();
  griddep_launch_dependents();
  const uint32_t tmem = *s_tmem;
  int rounds_issued = 0;  // MMA warp: accumulator rounds committed
  // Every CTA reads the same hidden rows: CTA c walks the K stages starting at
  // stage c mod NS, so at any moment about NC / NS CTAs (not all of them) load
  // the same hidden lines from L2.  Each logit's sum over K changes order only.
  const int k_rot = c % p.NS;

  // ======================= phase A: logits + slice statistics =============
  if (warp == 0) {
    const bool leader = elect_one();
    const uint64_t pol_w = l2_policy_evict_first();
    const uint64_t pol_h = l2_policy_evict_last();
    const uint32_t hk = p.Ncols * 128;  // hidden bytes per k-chunk
    uint32_t w_issued = 0, h_issued = 0;
    // Ring slots and parities advance by counters (no per-stage divisions).
    int ws = 0, hs = 0;
    uint32_t wph = 1, hph = 1;
    bool ok = true;
    int tdone = 0;
    for (int r = 0; ok && r < p.nrounds && tdone < ntiles; ++r) {
      const int nt = min(p.round_tiles[r], ntiles - tdone);
      int ks = k_rot;
      for (int it = 0; ok && it < p.NS; ++it) {
        const int c0 = ks * p.KG;
        const int nch = min(p.KG, p.KC - c0);
        const bool box3 = (nch == p.KG) && (c0 + p.KG <= p.KCF);
        if (++ks == p.NS) ks = 0;
        ok = warp_wait(&h_empty[hs], hph, s_abort);
        if (!ok) break;
        {
          uint8_t *dst = h_ring + hs * L.h_slot;
          if (leader) {
            mbar_arrive_expect_tx(&h_full[hs], nch * hk);
            if (box3) {
              tma_load_3d(dst, &tm_h3, 0, 0, c0, &h_full[hs], pol_h);
            } else {
              for (int j = 0; j < nch; ++j)
                tma_load_2d(dst + j * hk, &tm_h2, (c0 + j) * kKChunk, 0, &h_full[hs], pol_h);
            }
          }
          ++h_issued;
          if (++hs == p.HS) { hs = 0; hph ^= 1u; }
        }
        for (int j = 0; j < nt; ++j) {
          ok = warp_wait(&w_empty[ws], wph, s_abort);
          if (!ok) break;
          uint8_t *dst = w_ring + ws * L.w_slot;
          const int row0 = v_lo + (tdone + j) * kTileV;
          if (short_last && tdone + j == ntiles - 1) {
            // Partial last tile: BRS-row boxes (BRS a multiple of 8), the k-chunks
            // packed at BRS * 128-byte strides: one 3-D box per stage when it
            // holds KG full chunks (small 2-D boxes stream far slower).  The
            // slot's remaining rows feed accumulator lanes that are never read.
            if (leader) {
              mbar_arrive_expect_tx(&w_full[ws], nch * p.BRS * 128);
              if (box3) {
                tma_load_3d(dst, &tm_w3s, 0, row0, c0, &w_full[ws], pol_w);
              } else {
                for (int jj = 0; jj < nch; ++jj)
                  tma_load_2d(dst + jj * p.BRS * 128, &tm_w2s, (c0 + jj) * kKChunk, row0, &w_full[ws], pol_w);
              }
            }
          } else if (leader) {
            mbar_arrive_expect_tx(&w_full[ws], nch * kWChunkBytes);
            if (box3) {
              tma_load_3d(dst, &tm_w3, 0, row0, c0, &w_full[ws], pol_w);
            } else {
              for (int jj = 0; jj < nch; ++jj)
                tma_load_2d(dst + jj * kWChunkBytes, &tm_w2, (c0 + jj) * kKChunk, row0, &w_full[ws], pol_w);
            }
          }
          ++w_issued;
          if (++ws == p.WS) { ws = 0; wph ^= 1u; }
        }
      }
      tdone += nt;
    }
    if (!ok && leader) {
      // Every copy issued must land before the CTA's shared memory goes away.
      for (uint32_t j = (w_issued > (uint32_t)p.WS ? w_issued - p.WS : 0); j < w_issued; ++j)
        mbar_wait_unabortable(&w_full[j % p.WS], (j / p.WS) & 1);
      for (uint32_t j = (h_issued > (uint32_t)p.HS ? h_issued - p.HS : 0); j < h_issued; ++j)
        mbar_wait_unabortable(&h_full[j % p.HS], (j / p.HS) & 1);
    }
  } else if (warp == 1) {
    const bool leader = elect_one();
    int ws = 0, hs = 0;
    uint32_t wph = 0, hph = 0;
    int tdone = 0;
    // (an expired wait of the CTA ends the loops: the results are void.  The round's
    // commit still comes: teardown waits for it before the tensor memory goes away.)
    bool ok = true;
    for (int r = 0; ok && r < p.nrounds && tdone < ntiles; ++r) {
      const int nt = min(p.round_tiles[r], ntiles - tdone);
      const int buf = r & 1;
      // The half's previous round has been read.
      if (r > 1) ok = warp_wait(&acc_empty[buf], ((r >> 1) - 1) & 1, s_abort);
      tc_fence_after();
      int ks = k_rot;
      for (int it = 0; ok && it < p.NS; ++it) {
        const int nch = min(p.KG, p.KC - ks * p.KG);
        if (++ks == p.NS) ks = 0;
        ok = warp_wait(&h_full[hs], hph, s_abort);
        tc_fence_after();
        const uint32_t h_addr = smem_u32(h_ring + hs * L.h_slot);
        for (int j = 0; j < nt; ++j) {
          ok = ok && warp_wait(&w_full[ws], wph, s_abort);
          if (!ok) break;
          tc_fence_after();
          const uint32_t w_addr = smem_u32(w_ring + ws * L.w_slot);
          // k-chunk stride in the slot: a full tile's chunks are 16 KB apart,
          // the short last tile's are packed (BRS rows each).
          const uint32_t w_chunk = (short_last && tdone + j == ntiles - 1) ? static_cast<uint32_t>(p.BRS * 128)
                                                                          : static_cast<uint32_t>(kWChunkBytes);
          const uint32_t d_tmem = tmem + static_cast<uint32_t>(buf * kHalfCols + j * p.Ncols);
          for (int jj = 0; jj < nch; ++jj) {
            // Each operand's descriptor is built once per k-chunk; a K step of
            // 16 adds 32 bytes, 2 in the descriptor's address field.
            const uint64_t da = smem_desc_sw128(w_addr + jj * w_chunk);
            const uint64_t db = smem_desc_sw128(h_addr + jj * p.Ncols * 128);
#pragma unroll
            for (int k16 = 0; k16 < kKChunk / 16; ++k16)
              if (leader) tc_mma_f16(d_tmem, da + 2u * k16, db + 2u * k16, p.idesc, (it | jj | k16) != 0);
          }
          if (leader) tc_commit(&w_empty[ws]);
          if (++ws == p.WS) { ws = 0; wph ^= 1u; }
        }
        if (leader) tc_commit(&h_empty[hs]);
        if (++hs == p.HS) { hs = 0; hph ^= 1u; }
      }
      if (leader) tc_commit(&acc_full[buf]);
      ++rounds_issued;
      tdone += nt;
    }
  } else {
    // ---- epilogue warps: slice statistics per row, logits of sampled rows ----
    const int et = tid - 64;             // 0 .. kEpiThreads - 1
    const int ew = warp - 2;             // 0 .. kEpiWarps - 1
    const int q4 = warp & 3;             // TMEM lane quarter this warp may access
    const int part = ew >> 2;            // which of the quarter's two warps
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    float *T = reinterpret_cast<float *>(smem + L.off_tbuf + ew * kTBufBytes);
    clear_exchange(p.c, c * kEpiThreads + et, p.c.NC * kEpiThreads);
    setup_rows<kEpiThreads>(p.c, p.Ncols, seqs, rows, et);
    // The quarter's two warps take the (tile, 16-row block) items in turn; each
    // keeps running statistics of every block, in shared memory (one copy of
    // the block's code, whatever the row count).
    const int nblk = p.Ncols / kBlk;
    BlkStat *all_stats = reinterpret_cast<BlkStat *>(smem + L.off_stat);
    BlkStat *stats = all_stats + ew * nblk;
    for (int bk = 0; bk < nblk; ++bk) blk_init(stats[bk], lane);
    __syncwarp();
    int tdone = 0;
    for (int r = 0; r < p.nrounds && tdone < ntiles; ++r) {
      const int nt = min(p.round_tiles[r], ntiles - tdone);
      const int buf = r & 1;
      if (!mbar_wait(&acc_full[buf], (r >> 1) & 1, s_abort)) atomicOr(p.c.status, SPADE_DEV_TIMEOUT);
      tc_fence_after();
      for (int j = 0; j < nt; ++j) {
        const int t = tdone + j;
        const int v0 = v_lo + t * kTileV + q4 * 32;
        if (v0 >= v_hi) break;  // the slice ends before this quarter of its last tile
        const uint32_t col = tmem + lane_base + static_cast<uint32_t>(buf * kHalfCols + j * p.Ncols);
#pragma unroll 1
        for (int bk = (t * nblk + part) & 1; bk < nblk; bk += 2) {
          uint32_t raw[kBlk];
          load_block(col + bk * kBlk, raw);
          tmem_wait_ld();
          stat_block(p.c, raw, bk * kBlk, v0, v_hi, rows, T, lane, stats[bk]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
      tdone += nt;
    }
    fence_proxy_async();  // the draws read the stored logits by bulk copies
    // Merge the warps' statistics and publish this CTA's slice partials.
    named_bar(1, kEpiThreads);
    publish_slice(p.c, all_stats, nblk, c, et);
  }
  if (*s_abort) atomicOr(p.c.status, SPADE_DEV_TIMEOUT);

  // ======================= decisions, commit, draws =========================
  if constexpr (kCluster) {
    block_sync();
    cluster_sync();
  } else if (!grid_barrier(p.c.bar, p.c.NC)) {
    if (tid == 0) atomicOr(p.c.status, SPADE_DEV_TIMEOUT);
  }
  // (the rings are idle: the last round's accumulators were complete)
  rows_phase(p.c, *reinterpret_cast<RowsSmem *>(smem), seqs, rows, c, p.c.NC);

  // ---- teardown: every TMEM access above has completed --------------------
  tc_fence_before();
  block_sync();
  if (warp == 1) {
    // No MMA may still write TMEM when it is released (matters only after an
    // expired wait; otherwise the epilogue already consumed the last round).
    if (lane == 0)
      for (int r = max(0, rounds_issued - 2); r < rounds_issued; ++r)
        mbar_wait_unabortable(&acc_full[r & 1], (r >> 1) & 1);
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// Rounds of one CTA's `tiles` vocabulary tiles: as few as let a round's
// accumulators (Ncols columns each) fit half of the tensor memory -- every round
// reads the hidden rows once more -- of nearly equal sizes, the larger first.
// (3, 2, 2 tiles of a 7-tile slice at 72 rows; 3, 3, 1 ends with less statistics
// to take after the stream, but its one-tile round streams slower: the copies
// end at 168 us instead of 163.)
static bool plan_rounds(int tiles, int Ncols, int *round_tiles, int *nrounds) {
  const int fit = kHalfCols / Ncols;
  if (fit <= 0) return false;
  const int n = (tiles + fit - 1) / fit;
  if (n > kMaxRounds) return false;
  for (int r = 0; r < n; ++r) round_tiles[r] = tiles / n + (r < tiles % n ? 1 : 0);
  *nrounds = n;
  return true;
}

struct Plan {
  int T, NC, Ncols, Rs;
};

static Plan make_plan(int R, int V, int sms) {
  Plan pl;
  pl.T = (V + kTileV - 1) / kTileV;
  pl.NC = pl.T < sms ? pl.T : sms;
  if (pl.NC > kMaxNC) pl.NC = kMaxNC;
  pl.Ncols = (R + 15) / 16 * 16;
  pl.Rs = (R + 7) / 8 * 8;
  return pl;
}

// Slices are V/NC rows (floor or ceil); returns the tiles of the longest slice
// and the box rows (multiple of 8, < 128) that cover every partial last tile,
// or 128 when no slice ends in a tile short enough to be worth a short box.
static void slice_shape(int V, int NC, int *tiles_max, int *brs) {
  const int lmin = V / NC, lmax = lmin + (V % NC ? 1 : 0);
  *tiles_max = (lmax + kTileV - 1) / kTileV;
  int last = 0;
  for (int L : {lmin, lmax}) {
    const int rows = L - ((L + kTileV - 1) / kTileV - 1) * kTileV;
    if (rows < kTileV && rows > last) last = rows;
  }
  *brs = last == 0 ? kTileV : (last + 7) / 8 * 8;
}

// Whether the one-launch form takes the call: at most 256 rows (one MMA's N), at most
// 32 tiles per SM, and tiles x rows (rounded up to 8) within 512 accumulator columns
// (on 152 SMs 256 rows up to 32000 entries, 128 at 64000, 72 at 128256, 64 at 152064).
// The kernel's rounds would run with more, but CTA pairs, which stream the hidden
// rows half as often, are faster there (us, pairs / one launch, no row sampled and
// all: 80 rows x 4096 x 128256 161 / 164 and 190 / 193, 128 rows 165 / 179 and 203 / 223,
// 256 rows 199 / 230 and 254 / 296; 72 rows x 5120 x 152064 236 / 237 and 269 / 275; 136 rows x
// 4096 x 64000 92 / 121 and 108 / 138).  Top-p needs this form: the search's bins are
// laid out for it only.
static bool one_launch(int R, int V, int sms) {
  if (R > kMaxRes) return false;
  const Plan pl = make_plan(R, V, sms);
  int tiles = 0, brs = 0;
  slice_shape(V, pl.NC, &tiles, &brs);
  if (tiles > kMaxTilesPerCta) return false;
  int used = 0, done = 0;
  while (done < tiles) {
    const int fit = (kTmemCols - used) / pl.Ncols;
    if (fit <= 0) return false;
    const int n = fit < tiles - done ? fit : tiles - done;
    used += n * pl.Rs;
    done += n;
  }
  return used <= kTmemCols;
}

// Workspace: barrier words, slice partials, draft logits, merged statistics,
// share masses, nucleus bins (one launch only), logits of the rows of sampled
// sequences (every row may be one; rows of greedy sequences are never touched).
struct WsLayout {
  bool two_launches;
  int NC, ldl;
  size_t pstat, ldraft, gstat, zpart, nhist, logits, end;
};
static WsLayout ws_layout(int B, int R, int V, int sms) {
  WsLayout L{};
  L.two_launches = !one_launch(R, V, sms);
  L.NC = L.two_launches ? pair_slices(V, sms) : make_plan(R, V, sms).NC;
  L.ldl = static_cast<int>(round_up(V, 4));
  const size_t rows = static_cast<size_t>(R);
  size_t off = kBarBytes;
  L.pstat = off;
  off += round_up(rows * L.NC * 16, 256);
  L.ldraft = off;
  off += round_up(rows * 4, 256);
  L.gstat = off;
  off += round_up(rows * 16, 256);
  L.zpart = off;
  off += round_up(static_cast<size_t>(2) * B * kMaxGroup * 8, 256);
  L.nhist = off;
  if (!L.two_launches) off += round_up(static_cast<size_t>(kNucRounds) * kMaxGroup * rows * kNucBins * 4, 256);
  L.logits = off;
  off += round_up(rows * L.ldl * 4, 256);
  L.end = off;
  return L;
}

struct Maps {
  CUtensorMap w3, w2, w2s, w3s, h3, h2;
};

// Fills the plan-dependent fields of `p` for the one-launch form over the rows
// of `hidden` ([R, H]) and encodes its tensor maps.
static spade_status prepare(Params &p, const void *hidden, const void *w_lm, int H, int sms, Maps &m) {
  const int R = p.c.R, V = p.c.V;
  const Plan pl = make_plan(R, V, sms);
  p.T = pl.T;
  p.Ncols = pl.Ncols;
  p.KC = (H + kKChunk - 1) / kKChunk;
  p.KCF = H / kKChunk;
  int tiles_max = 0;
  slice_shape(V, pl.NC, &tiles_max, &p.BRS);
  if (!plan_rounds(tiles_max, pl.Ncols, p.round_tiles, &p.nrounds))
    return fail(SPADE_ERR_SHAPE, "%d rows x %d tiles per SM do not fit the accumulator rounds", R, tiles_max);
  p.idesc = idesc_bf16_f32(kTileV, pl.Ncols);
  p.HS = 3;
  p.KG = 2;  // two k-chunks per stage (32 KB W boxes) while the rings fit
  for (;;) {
    Params probe = p;
    probe.WS = 0;
    const int fixed = smem_layout(probe).total;
    p.WS = (kSmemMax - 1024 - fixed) / (p.KG * kWChunkBytes);  // 1 KB for static shared memory
    if (p.WS > 8) p.WS = 8;
    if (p.WS >= 4 || p.KG == 1) break;
    p.KG = 1;
  }
  if (p.WS < 2) return fail(SPADE_ERR_SHAPE, "shared memory too small for R = %d", R);
  // After the stream the rows phase works in the rings.
  const size_t rings = static_cast<size_t>(smem_layout(p).off_bar);
  const size_t items = R < kWarps ? kWarps : R;  // rows or parts of rows that the nucleus search lists, at most
  const size_t pool0 = offsetof(RowsSmem, pool);
  if (rings < (p.c.top_p ? pool0 + items * kPoolPerRow : kRowsBytesPlain))
    return fail(SPADE_ERR_SHAPE, "shared memory too small for R = %d", R);
  p.c.pool = static_cast<int>(rings - pool0);
  p.NS = (p.KC + p.KG - 1) / p.KG;

  // 2-D views (one k-chunk per box, zero fill past H) serve a ragged last
  // k-chunk; 3-D views fetch KG full k-chunks.
  const uint64_t pitch = static_cast<uint64_t>(H) * 2;
  if (!encode_tmap_bf16_sw128(&m.w2, w_lm, H, V, pitch, kKChunk, kTileV) ||
      !encode_tmap_bf16_sw128(&m.w2s, w_lm, H, V, pitch, kKChunk, p.BRS) ||
      !encode_tmap_bf16_sw128(&m.h2, hidden, H, R, pitch, kKChunk, pl.Ncols))
    return SPADE_ERR_CUDA;
  if (p.KCF >= 1) {
    if (!encode_tmap_rows_by_slab(&m.w3, w_lm, V, H, kTileV, p.KG) || !encode_tmap_rows_by_slab(&m.w3s, w_lm, V, H, p.BRS, p.KG) ||
        !encode_tmap_rows_by_slab(&m.h3, hidden, R, H, pl.Ncols, p.KG))
      return SPADE_ERR_CUDA;
  } else {
    m.w3 = m.w2;  // never used: every stage takes the 2-D path
    m.w3s = m.w2s;
    m.h3 = m.h2;
  }
  return SPADE_OK;
}

// Grids of at most this many CTAs (vocabularies up to 1024 entries) run as one
// cluster: its CTAs are resident together without the cooperative attribute, which
// costs 2.7 us between dependent launches, and meet at the cluster's hardware
// barrier instead of the grid's in L2 (2.0-2.8 us).  5 rows x 512 x 1024: 16.4 ->
// 11.8 us.  (8: the cluster size that every device of this kind takes.)
constexpr int kMaxCluster = 8;

// Whether the device takes such a cluster (asked once per device and size, with
// the most shared memory that a call may need; a failed question is asked again).
static bool cluster_fits(cudaLaunchConfig_t cfg, int n) {
  static std::atomic<signed char> known[kMaxDevices][kMaxCluster + 1];  // 0: not asked, 1: yes, -1: no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev >= kMaxDevices) return false;
  signed char k = known[dev][n].load(std::memory_order_relaxed);
  if (k == 0) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = n;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.dynamicSmemBytes = kSmemMax - 1024;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int active = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&active, verify_accept_kernel<true>, &cfg);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    k = active > 0 ? 1 : -1;
    known[dev][n].store(k, std::memory_order_relaxed);
  }
  return k > 0;
}

static spade_status launch(const Params &p, const Maps &m, cudaStream_t stream) {
  static OncePerDevice once;
  const cudaError_t es = set_max_smem(once, kSmemMax - 1024, verify_accept_kernel<false>, verify_accept_kernel<true>);
  if (es != cudaSuccess) return cuda_fail(es, "cudaFuncSetAttribute(verify_accept)");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.c.NC);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem_layout(p).total;
  cfg.stream = stream;
  // Cooperative or one cluster: the CTAs meet at barriers.  Programmatic: a CTA
  // starts as soon as the previous kernel has left its SM (it waits for that
  // kernel's end before it reads anything).
  const bool cluster = p.c.NC <= kMaxCluster && cluster_fits(cfg, p.c.NC);
  cudaLaunchAttribute attr[2];
  if (cluster) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.c.NC;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, cluster ? verify_accept_kernel<true> : verify_accept_kernel<false>, p, m.w3, m.w2, m.w2s, m.w3s, m.h3, m.h2);
  if (e != cudaSuccess) return cuda_fail(e, "verify_accept launch");
  return SPADE_OK;
}

}  // namespace accept
}  // namespace spade

using namespace spade;

extern "C" int32_t spade_accept_launches(int32_t B, int32_t R, int32_t H, int32_t V) {
  if (B <= 0 || R < B || H <= 0 || V <= 0) return 0;
  int sms = 0;
  if (device_info(&sms, nullptr) != SPADE_OK) return 0;
  return accept::one_launch(R, V, sms) ? 1 : 2;
}

extern "C" size_t spade_accept_workspace_size(int32_t B, int32_t R, int32_t H, int32_t V) {
  if (B <= 0 || R < B || H <= 0 || V <= 0) return 0;
  int sms = 0;
  if (device_info(&sms, nullptr) != SPADE_OK) return 0;
  return accept::ws_layout(B, R, V, sms).end;
}

extern "C" spade_status spade_accept_stats_layout(int32_t B, int32_t R, int32_t H, int32_t V,
                                                  size_t *row_stats_offset, size_t *draft_logit_offset,
                                                  int32_t *replica_stride) {
  if (!row_stats_offset || !draft_logit_offset || !replica_stride)
    return fail(SPADE_ERR_INVALID_ARG, "spade_accept_stats_layout: null output pointer");
  if (B <= 0 || R < B || H <= 0 || V <= 0)
    return fail(SPADE_ERR_INVALID_ARG, "spade_accept_stats_layout: bad sizes B=%d R=%d H=%d V=%d", B, R, H, V);
  int sms = 0;
  const spade_status st = device_info(&sms, nullptr);
  if (st != SPADE_OK) return st;
  const accept::WsLayout L = accept::ws_layout(B, R, V, sms);
  *row_stats_offset = L.gstat;
  *draft_logit_offset = L.ldraft;
  *replica_stride = R;
  return SPADE_OK;
}

namespace spade {
namespace accept {
struct CommitArgs {
  void *k_cache, *v_cache;
  int32_t *ctx_lens;
  int Hkv, D, cap;
  const int32_t *block_table;  // paged pools when non-null
  int page_size, max_pages, num_pages;
};
static spade_status verify_accept_impl(const void *hidden, const void *w_lm,
                                       const int32_t *draft_tokens, const float *draft_probs,
                                       const float *uniforms, const int32_t *mode,
                                       const int32_t *cu_q, const int32_t *n_draft,
                                       int32_t *accepted_len, int32_t *next_token, int32_t B,
                                       int32_t R, int32_t H, int32_t V, void *workspace,
                                       size_t workspace_bytes, int32_t *status,
                                       spade_stream_t stream, const CommitArgs *cm,
                                       const float *temperature = nullptr,
                                       const float *top_p = nullptr) {
  using namespace accept;
  if (!hidden || !w_lm || !uniforms || !mode || !cu_q || !n_draft || !accepted_len ||
      !next_token || !status || (R > B && !draft_tokens))
    return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept: null pointer argument");
  if (B <= 0 || R < B || H <= 0 || V <= 0)
    return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept: bad sizes B=%d R=%d H=%d V=%d", B, R, H, V);
  if (H % 8) return fail(SPADE_ERR_SHAPE, "hidden size %d must be a multiple of 8", H);
  if (R > kMaxR) return fail(SPADE_ERR_SHAPE, "R = %d verify rows exceed %d per call", R, kMaxR);
  if (B > kMaxB) return fail(SPADE_ERR_SHAPE, "B = %d sequences exceed %d per call", B, kMaxB);
  if (!aligned(hidden, 16) || !aligned(w_lm, 16))
    return fail(SPADE_ERR_INVALID_ARG, "hidden and w_lm must be 16-byte aligned");
  int sms = 0;
  spade_status st = device_info(&sms, nullptr);
  if (st != SPADE_OK) return st;

  int tiles = 0, brs = 0;
  slice_shape(V, make_plan(R, V, sms).NC, &tiles, &brs);
  if (tiles > kMaxTilesPerCta)
    return fail(SPADE_ERR_SHAPE, "vocabulary %d needs %d tiles per SM (max %d)", V, tiles, kMaxTilesPerCta);
  const WsLayout L = ws_layout(B, R, V, sms);
  if (top_p && L.two_launches)
    return fail(SPADE_ERR_SHAPE, "top-p needs the one-launch form: R = %d rows x V = %d exceed it", R, V);
  if (!workspace || workspace_bytes < L.end || !aligned(workspace, 256))
    return fail(SPADE_ERR_WORKSPACE, "accept workspace needs %zu bytes, 256-byte aligned (got %zu)",
                L.end, workspace_bytes);
  uint8_t *ws = static_cast<uint8_t *>(workspace);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);

  Params p{};
  Call &c = p.c;
  c.draft_tokens = draft_tokens;
  c.draft_probs = draft_probs;
  c.temperature = temperature;
  c.top_p = top_p;
  c.qvec = draft_probs != nullptr && aligned(draft_probs, 16) && V % 4 == 0;
  c.uniforms = uniforms;
  c.mode = mode;
  c.cu_q = cu_q;
  c.n_draft = n_draft;
  c.accepted_len = accepted_len;
  c.next_token = next_token;
  c.status = status;
  c.B = B;
  c.R = R;
  c.V = V;
  c.NC = L.NC;
  c.ldl = L.ldl;
  c.bar = reinterpret_cast<unsigned *>(ws);
  c.pstat = reinterpret_cast<float4 *>(ws + L.pstat);
  c.ldraft = reinterpret_cast<float *>(ws + L.ldraft);
  c.gstat = reinterpret_cast<float4 *>(ws + L.gstat);
  c.zpart = reinterpret_cast<unsigned long long *>(ws + L.zpart);
  c.nhist = reinterpret_cast<unsigned *>(ws + L.nhist);
  c.logits = reinterpret_cast<float *>(ws + L.logits);
  if (cm) {
    c.kc = static_cast<uint4 *>(cm->k_cache);
    c.vc = static_cast<uint4 *>(cm->v_cache);
    c.ctx_lens = cm->ctx_lens;
    c.Hkv = cm->Hkv;
    c.Dk = cm->D;
    c.cap = cm->cap;
    c.block_table = cm->block_table;
    c.page_size = cm->page_size;
    c.max_pages = cm->max_pages;
    c.num_pages = cm->num_pages;
  }
  if (L.two_launches) {
    c.pool = kPieceBytes;  // (no nucleus search on this path)
    st = launch_lm_head_pairs(c, hidden, w_lm, H, s);
    return st != SPADE_OK ? st : launch_accept_rows(c, sms, s);
  }
  Maps m;
  st = prepare(p, hidden, w_lm, H, sms, m);
  return st != SPADE_OK ? st : launch(p, m, s);
}
}  // namespace accept
}  // namespace spade

extern "C" spade_status spade_verify_accept(const void *hidden, const void *w_lm,
                                            const int32_t *draft_tokens, const float *draft_probs,
                                            const float *uniforms, const int32_t *mode,
                                            const int32_t *cu_q, const int32_t *n_draft,
                                            int32_t *accepted_len, int32_t *next_token, int32_t B,
                                            int32_t R, int32_t H, int32_t V, void *workspace,
                                            size_t workspace_bytes, int32_t *status,
                                            spade_stream_t stream) {
  return accept::verify_accept_impl(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q,
                                    n_draft, accepted_len, next_token, B, R, H, V, workspace,
                                    workspace_bytes, status, stream, nullptr);
}

extern "C" spade_status spade_verify_accept_commit(
    const void *hidden, const void *w_lm, const int32_t *draft_tokens, const float *draft_probs,
    const float *uniforms, const int32_t *mode, const int32_t *cu_q, const int32_t *n_draft,
    int32_t *accepted_len, int32_t *next_token, void *k_cache, void *v_cache, int32_t *ctx_lens,
    int32_t B, int32_t R, int32_t H, int32_t V, int32_t Hkv, int32_t D, int32_t cap,
    void *workspace, size_t workspace_bytes, int32_t *status, spade_stream_t stream) {
  if (!k_cache || !v_cache || !ctx_lens)
    return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_commit: null cache or ctx_lens pointer");
  if (Hkv <= 0 || D <= 0 || cap <= 0)
    return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_commit: non-positive cache size");
  if (D % 8) return fail(SPADE_ERR_SHAPE, "spade_verify_accept_commit: D = %d must be a multiple of 8", D);
  if (!aligned(k_cache, 16) || !aligned(v_cache, 16))
    return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_commit: caches must be 16-byte aligned");
  const accept::CommitArgs cm{k_cache, v_cache, ctx_lens, Hkv, D, cap, nullptr, 0, 0, 0};
  return accept::verify_accept_impl(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q,
                                    n_draft, accepted_len, next_token, B, R, H, V, workspace,
                                    workspace_bytes, status, stream, &cm);
}

extern "C" spade_status spade_verify_accept_commit_paged(
    const void *hidden, const void *w_lm, const int32_t *draft_tokens, const float *draft_probs,
    const float *uniforms, const int32_t *mode, const int32_t *cu_q, const int32_t *n_draft,
    int32_t *accepted_len, int32_t *next_token, void *k_pool, void *v_pool, const int32_t *block_table,
    int32_t *ctx_lens, int32_t B, int32_t R, int32_t H, int32_t V, int32_t Hkv, int32_t D, int32_t page_size,
    int32_t num_pages, int32_t max_pages, void *workspace, size_t workspace_bytes, int32_t *status,
    spade_stream_t stream) {
  if (!k_pool || !v_pool || !block_table || !ctx_lens)
    return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_commit_paged: null pool, table or ctx_lens pointer");
  if (Hkv <= 0 || D <= 0 || page_size <= 0 || num_pages <= 0 || max_pages <= 0)
    return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_commit_paged: non-positive size");
  if (D % 8) return fail(SPADE_ERR_SHAPE, "spade_verify_accept_commit_paged: D = %d must be a multiple of 8", D);
  if (static_cast<int64_t>(max_pages) * page_size >= (int64_t(1) << 31))
    return fail(SPADE_ERR_CAPACITY, "max_pages * page_size exceeds 2^31");
  if (!aligned(k_pool, 16) || !aligned(v_pool, 16))
    return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_commit_paged: pools must be 16-byte aligned");
  const accept::CommitArgs cm{k_pool, v_pool, ctx_lens, Hkv, D, max_pages * page_size, block_table,
                              page_size, max_pages, num_pages};
  return accept::verify_accept_impl(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q,
                                    n_draft, accepted_len, next_token, B, R, H, V, workspace,
                                    workspace_bytes, status, stream, &cm);
}

extern "C" spade_status spade_verify_accept_temperature(
    const void *hidden, const void *w_lm, const int32_t *draft_tokens, const float *draft_probs,
    const float *uniforms, const int32_t *mode, const float *temperature, const int32_t *cu_q,
    const int32_t *n_draft, int32_t *accepted_len, int32_t *next_token, int32_t B, int32_t R, int32_t H,
    int32_t V, void *workspace, size_t workspace_bytes, int32_t *status, spade_stream_t stream) {
  if (!temperature) return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_temperature: null temperature");
  return accept::verify_accept_impl(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
                                    accepted_len, next_token, B, R, H, V, workspace, workspace_bytes, status,
                                    stream, nullptr, temperature);
}

extern "C" spade_status spade_verify_accept_sampling(
    const void *hidden, const void *w_lm, const int32_t *draft_tokens, const float *draft_probs,
    const float *uniforms, const int32_t *mode, const float *temperature, const float *top_p,
    const int32_t *cu_q, const int32_t *n_draft, int32_t *accepted_len, int32_t *next_token, void *k_cache,
    void *v_cache, int32_t *ctx_lens, int32_t B, int32_t R, int32_t H, int32_t V, int32_t Hkv, int32_t D,
    int32_t cap, void *workspace, size_t workspace_bytes, int32_t *status, spade_stream_t stream) {
  const bool commit = k_cache || v_cache || ctx_lens;
  if (commit) {
    if (!k_cache || !v_cache || !ctx_lens)
      return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_sampling: give all of k_cache, v_cache, ctx_lens or none");
    if (Hkv <= 0 || D <= 0 || cap <= 0)
      return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_sampling: non-positive cache size");
    if (D % 8) return fail(SPADE_ERR_SHAPE, "spade_verify_accept_sampling: D = %d must be a multiple of 8", D);
    if (!aligned(k_cache, 16) || !aligned(v_cache, 16))
      return fail(SPADE_ERR_INVALID_ARG, "spade_verify_accept_sampling: caches must be 16-byte aligned");
  }
  const accept::CommitArgs cm{k_cache, v_cache, ctx_lens, Hkv, D, cap, nullptr, 0, 0, 0};
  return accept::verify_accept_impl(hidden, w_lm, draft_tokens, draft_probs, uniforms, mode, cu_q, n_draft,
                                    accepted_len, next_token, B, R, H, V, workspace, workspace_bytes, status,
                                    stream, commit ? &cm : nullptr, temperature, top_p);
}
