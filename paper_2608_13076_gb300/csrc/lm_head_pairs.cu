// lm_head_pairs.cu -- first launch of the two-launch LM head (calls that the
// one-launch form does not take, see one_launch()): logits o = g(x_L) of every verify
// row against the vocabulary (Sec. III-A), kept as per-slice softmax statistics,
// and stored for the rows that a sampled sequence may draw from.
//
// Design (GB300): bound by the tensor pipe at R ~ 400 rows (0.8 flop per byte of
// W and row), so the MMAs run on CTA pairs (clusters of two, tcgen05
// cta_group::2): one MMA of M = 256 takes 128 W rows from each CTA's shared
// memory and splits each N-chunk's hidden rows between the two, so an SM
// receives 16 KB of W and half of the hidden rows per k-chunk of 64.
//  * Each CTA owns a contiguous vocabulary slice, cut into tiles of equal height
//    (at most 128 rows): the pair's MMA covers one tile of each.
//  * Rows up to 256 leave room for two accumulators, and the statistics of a
//    tile run under the next one's MMAs; more rows fill tensor memory, and
//    sixteen statistics warps empty it between tiles.
//  * The rows of sampled sequences store their fp32 logits (coalesced 128-byte
//    rows straight from the accumulators).  A draw then reads one stored row
//    instead of streaming W again: 118 MB written against 1.56 GB re-read at
//    389 rows x 152064 entries.
#include "accept_launch.h"

namespace spade {
namespace accept {

constexpr int kMaxStages = 8;
// Four statistics warps per tensor-memory lane quarter: the statistics of more
// than 256 rows do not run under the next tile's MMAs, and eight warps leave
// their latencies uncovered (this launch at 389 rows x 5120 x 152064: 405 us with
// eight, 380 with sixteen and blocks reduced in pairs; 343 without statistics.
// Blocks held in registers, so that the next tile's MMAs start under them, gave
// nothing more: the launch is then short of power, 1.4 kW, not of time).
constexpr int kPairWarps = 16;
constexpr int kPairEpi = 32 * kPairWarps;
constexpr int kPairThreads = 64 + kPairEpi;
constexpr int kParts = kPairWarps / 4;

struct PairParams {
  Call c;
  int KC;            // k-chunks of 64 (the last may be partial: zero-filled)
  int th;            // rows per tile and CTA
  int ntiles;        // tiles of the longest slice
  int Ncols;         // rows rounded up to 16
  int n0w, n1w;      // widths of the MMA N-chunks (n1w = 0: one chunk)
  int nacc;          // accumulators (2 when two fit)
  int stages;
  uint32_t idesc0, idesc1;
};

struct PairSmem {
  int stage, off_bar, off_misc, off_seq, off_rows, off_stat, off_tbuf, total;
};
__host__ __device__ inline PairSmem pair_layout(int Ncols, int stages) {
  PairSmem s;
  s.stage = kWChunkBytes + Ncols / 2 * 128;  // W rows, then this CTA's half of each N-chunk
  s.off_bar = stages * s.stage;
  s.off_misc = s.off_bar + (2 * kMaxStages + 4) * 8;
  s.off_seq = (s.off_misc + 16 + 15) & ~15;
  s.off_rows = s.off_seq + static_cast<int>(sizeof(SeqTable));
  s.off_stat = s.off_rows + row_table_bytes(Ncols, false);
  // A statistics warp keeps every kParts-th block of rows.
  const int per = (Ncols / kBlk + kParts - 1) / kParts;
  s.off_tbuf = (s.off_stat + kPairWarps * per * static_cast<int>(sizeof(BlkStat)) + 127) & ~127;
  s.total = s.off_tbuf + kPairWarps * kTBufBytes + 1024;
  return s;
}

// Vocabulary slice of CTA `rank` of pair j.  Pairs walk the k-chunks from different
// starts, so that not all of them load the same hidden lines from L2 at once:
// slice s from chunk 2 (s mod ns), as the one-launch form walks it with stages of two
// chunks (up to 80 rows; with one-chunk stages, above, it starts at another chunk).
// A pair has one order: it takes slices s and s + ns, which share it, so their logits
// are summed in the one-launch form's order, to the same bits.  Slices without such a
// partner pair up with their neighbours, and the second of the two takes the first's
// order (4 of 152 slices at H = 5120, 12 at 4096 and 8192, 20 at 12288, 76 at 20480).
__device__ __forceinline__ int pair_slice(int j, int rank, int nslices, int ns) {
  const int group = j / ns, i = j - group * ns, base = 2 * ns * group;
  const int both = max(0, min(nslices - base, 2 * ns) - ns);  // pairs (s, s + ns) of this group
  return i < both ? base + i + rank * ns : base + both + 2 * (i - both) + rank;
}

__global__ void __launch_bounds__(kPairThreads, 1) lm_head_pairs_kernel(
    const __grid_constant__ PairParams p, const __grid_constant__ CUtensorMap tm_w,
    const __grid_constant__ CUtensorMap tm_h0, const __grid_constant__ CUtensorMap tm_h1) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const PairSmem L = pair_layout(p.Ncols, p.stages);
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + L.off_bar);
  uint64_t *empty = full + kMaxStages;
  uint64_t *acc_full = empty + kMaxStages;  // [2]
  uint64_t *acc_empty = acc_full + 2;       // [2]
  volatile int *s_abort = reinterpret_cast<volatile int *>(smem + L.off_misc);
  uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L.off_misc + 8);
  const RowTables rows = row_tables(smem + L.off_rows, p.Ncols, false);

  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  const int ns = (p.KC + 1) / 2;
  const int c = pair_slice(blockIdx.x >> 1, rank, p.c.NC, ns);
  const int v_lo = static_cast<int>(static_cast<int64_t>(c) * p.c.V / p.c.NC);
  const int v_hi = static_cast<int>(static_cast<int64_t>(c + 1) * p.c.V / p.c.NC);
  // Both CTAs of a pair walk p.ntiles tiles (a slice one row shorter may leave
  // its last tile without valid rows: its copies are still made, its statistics
  // are masked).
  const uint32_t stage_tx = static_cast<uint32_t>(p.th * 128 + p.Ncols / 2 * 128);  // bytes one CTA copies per stage

  // ---- set-up that reads no input ------------------------------------------
  if (tid == 0) {
    *s_abort = 0;
    for (int s = 0; s < p.stages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 2 * kPairWarps); }
    if (rank == 0)  // arm every stage's first use with both CTAs' bytes
      for (int s = 0; s < p.stages; ++s) mbar_arrive_expect_tx(&full[s], 2 * stage_tx);
    fence_mbar_init();
    tma_prefetch_desc(&tm_w);
    tma_prefetch_desc(&tm_h0);
    if (p.n1w) tma_prefetch_desc(&tm_h1);
  }
  if (warp == 1) {
    tmem_alloc_pair(s_tmem, kTmemCols);  // collective: the same columns in both SMs
    tmem_relinquish_pair();
  }
  tc_fence_before();
  block_sync();
  cluster_sync();  // both CTAs' barriers exist before either signals the other
  tc_fence_after();
  griddep_wait();
  griddep_launch_dependents();
  const uint32_t tmem = *s_tmem;
  const uint32_t h1_off = static_cast<uint32_t>(kWChunkBytes + p.n0w / 2 * 128);
  int tiles_issued = 0;
  const int k_rot = 2 * (pair_slice(blockIdx.x >> 1, 0, p.c.NC, ns) % ns);

  if (warp == 0) {
    // Both CTAs' copies of a stage complete on the even CTA's full barrier,
    // armed with the bytes of both before either CTA may issue them (at
    // set-up, then by the MMA warp as it takes the previous use).
    const bool leader = elect_one();
    const uint64_t pol_w = l2_policy_evict_first(), pol_h = l2_policy_evict_last();
    const uint32_t full0 = cluster_map(full, 0);
    const int hrow0 = static_cast<int>(rank) * (p.n0w / 2);
    const int hrow1 = p.n0w + static_cast<int>(rank) * (p.n1w / 2);
    uint32_t issued = 0, eph = 1;
    int s = 0;
    bool ok = true;
    for (int t = 0; ok && t < p.ntiles; ++t) {
      const int row0 = v_lo + t * p.th;
      int kc = k_rot;
      for (int it = 0; it < p.KC; ++it) {
        ok = warp_wait(&empty[s], eph, s_abort);
        if (!ok) break;
        uint8_t *dst = smem + s * L.stage;
        const uint32_t bar = full0 + 8u * s;
        const int kx = kc * kKChunk;
        if (leader) {
          tma_load_2d_pair(dst, &tm_w, kx, row0, bar, pol_w);
          tma_load_2d_pair(dst + kWChunkBytes, &tm_h0, kx, hrow0, bar, pol_h);
        }
        if (p.n1w) {
          if (leader) tma_load_2d_pair(dst + h1_off, &tm_h1, kx, hrow1, bar, pol_h);
        }
        ++issued;
        if (++kc == p.KC) kc = 0;
        if (++s == p.stages) { s = 0; eph ^= 1u; }
      }
    }
    // After an expired wait the even CTA drains the copies of both (its full
    // barriers count them); the odd CTA's shared memory stays alive until both
    // CTAs have reached the teardown.
    if (!ok && rank == 0 && leader) {
      const uint32_t n = p.stages;
      for (uint32_t j = (issued > n ? issued - n : 0); j < issued; ++j)
        if (!mbar_wait_unabortable(&full[j % n], (j / n) & 1)) break;  // (the odd CTA stopped before this stage)
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // Even CTA: M = 256 MMAs over both CTAs' stages; the stages are freed in
      // both CTAs by one multicast commit.  (An expired wait of the CTA ends the
      // MMAs: the results are void.  Every tile's commit still comes, as both
      // CTAs' teardown waits for the last ones.)
      const bool leader = elect_one();
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int t = 0; t < p.ntiles; ++t) {
        const int buf = p.nacc == 2 ? t & 1 : 0, use = p.nacc == 2 ? t >> 1 : t;
        const uint32_t d0 = tmem + static_cast<uint32_t>(buf * (kTmemCols / 2));
        const uint32_t d1 = d0 + static_cast<uint32_t>(p.n0w);
        if (ok && use > 0) {
          if (leader) mbar_wait_cluster(&acc_empty[buf], (use - 1) & 1, s_abort);
          __syncwarp();
        }
        tc_fence_after();
        for (int it = 0; ok && it < p.KC; ++it) {
          // (cta-scope wait: the copies' completion on this barrier orders them
          // for the MMAs issued after it, the odd CTA's included)
          ok = warp_wait(&full[s], ph, s_abort);
          if (!ok) break;
          // Arm the stage's next use now: its copies are issued only after this
          // use's commit frees the stage.
          if (leader) mbar_arrive_expect_tx(&full[s], 2 * stage_tx);
          tc_fence_after();
          const uint32_t base = smem_u32(smem + s * L.stage);
          const uint64_t da = smem_desc_sw128(base), db0 = smem_desc_sw128(base + kWChunkBytes);
          const uint64_t db1 = smem_desc_sw128(base + h1_off);
#pragma unroll
          for (int k16 = 0; k16 < kKChunk / 16; ++k16) {
            if (leader) tc_mma_f16_pair(d0, da + 2u * k16, db0 + 2u * k16, p.idesc0, (it | k16) != 0);
            if (p.n1w) {
              if (leader) tc_mma_f16_pair(d1, da + 2u * k16, db1 + 2u * k16, p.idesc1, (it | k16) != 0);
            }
          }
          if (leader) tc_commit_pair(&empty[s]);
          if (++s == p.stages) { s = 0; ph ^= 1u; }
        }
        if (leader) tc_commit_pair(&acc_full[buf]);
        ++tiles_issued;
      }
    } else {
      tiles_issued = p.ntiles;  // odd CTA: the even CTA's commits reach its acc_full too
    }
  } else {
    // ---- statistics warps ----
    const int et = tid - 64, ew = warp - 2, q4 = warp & 3, part = ew >> 2;
    const uint32_t lane_base = static_cast<uint32_t>(q4 * 32) << 16;
    float *T = reinterpret_cast<float *>(smem + L.off_tbuf + ew * kTBufBytes);
    clear_exchange(p.c, c * kPairEpi + et, p.c.NC * kPairEpi);
    setup_rows<kPairEpi>(p.c, p.Ncols, *reinterpret_cast<SeqTable *>(smem + L.off_seq), rows, et);
    const int nblk = p.Ncols / kBlk, per = (nblk + kParts - 1) / kParts;
    BlkStat *stats = reinterpret_cast<BlkStat *>(smem + L.off_stat) + ew * per;
    for (int j = 0; j < per; ++j) blk_init(stats[j], lane);
    __syncwarp();
    const uint32_t empty0 = cluster_map(acc_empty, 0);
    for (int t = 0; t < p.ntiles; ++t) {
      const int buf = p.nacc == 2 ? t & 1 : 0, use = p.nacc == 2 ? t >> 1 : t;
      if (!mbar_wait(&acc_full[buf], use & 1, s_abort)) atomicOr(p.c.status, SPADE_DEV_TIMEOUT);
      tc_fence_after();
      const int v0 = v_lo + t * p.th + q4 * 32;
      const int hi = min(v_hi, v_lo + (t + 1) * p.th);  // the tile's valid entries end here
      const uint32_t col = tmem + lane_base + static_cast<uint32_t>(buf * (kTmemCols / 2));
      if (v0 < hi) {
#pragma unroll 1
        for (int bk = part; bk < nblk; bk += kParts) {
          uint32_t raw[kBlk];
          load_block(col + bk * kBlk, raw);
          tmem_wait_ld();
          stat_block(p.c, raw, bk * kBlk, v0, hi, rows, T, lane, stats[bk / kParts]);
        }
      }
      // The accumulator is read: the MMA thread counts both CTAs' warps.
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0) mbar_arrive(&acc_empty[buf]);
        else mbar_arrive_cluster(empty0 + 8u * buf);
      }
    }
    // Merge the warps' statistics and publish this CTA's slice partials.
    named_bar(1, kPairEpi);
    const BlkStat *all = reinterpret_cast<const BlkStat *>(smem + L.off_stat);
    for (int n = et; n < p.c.R; n += kPairEpi) {
      const int bk = n / kBlk;
      float m = -INFINITY, z = 0.f;
      int idx = INT_MAX;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const BlkStat &st = all[((bk % kParts) * 4 + w) * per + bk / kParts];
        stat_merge(m, z, idx, st.m[n % kBlk], st.s[n % kBlk], st.i[n % kBlk]);
      }
      __stcg(&p.c.pstat[static_cast<size_t>(n) * p.c.NC + c], make_float4(m, z, __int_as_float(idx), 0.f));
    }
  }
  if (*s_abort) atomicOr(p.c.status, SPADE_DEV_TIMEOUT);

  // ---- teardown: every TMEM access above has completed --------------------
  tc_fence_before();
  block_sync();
  if (warp == 1) {
    if (lane == 0) {
      // No MMA may still write TMEM or read the other CTA's stages (matters
      // only after an expired wait: the statistics consumed the last tile).
      for (int t = max(0, tiles_issued - p.nacc); t < tiles_issued; ++t)
        mbar_wait_unabortable(&acc_full[p.nacc == 2 ? t & 1 : 0], (p.nacc == 2 ? t >> 1 : t) & 1);
    }
    __syncwarp();
  }
  // Both CTAs are done with the allocation, with each other's shared memory and with
  // each other's barriers.  (The cluster's barrier has no limit, and needs none: each
  // wait before it has one, so both CTAs come.  After an expired wait one of them may
  // come seconds after the other, which must not have left: its barriers are still
  // arrived on.)
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kTmemCols);
  }
}

int pair_slices(int V, int sms) {
  const int most = (sms < kMaxNC ? sms : kMaxNC) / 2;
  const int pairs = (V + 2 * kTileV - 1) / (2 * kTileV);
  return 2 * (pairs < most ? pairs : most);
}

spade_status launch_lm_head_pairs(const Call &c, const void *hidden, const void *w_lm, int H, cudaStream_t stream) {
  PairParams p{};
  p.c = c;
  p.KC = (H + kKChunk - 1) / kKChunk;
  p.Ncols = (c.R + 15) / 16 * 16;
  if (p.Ncols > kTmemCols) return fail(SPADE_ERR_SHAPE, "R = %d rows exceed %d", c.R, kTmemCols);
  const int lmax = (c.V + c.NC - 1) / c.NC;  // longest slice
  p.ntiles = (lmax + kTileV - 1) / kTileV;
  p.th = (lmax + p.ntiles - 1) / p.ntiles;
  p.n0w = p.Ncols > 256 ? (p.Ncols / 2 + 15) / 16 * 16 : p.Ncols;
  p.n1w = p.Ncols - p.n0w;
  p.nacc = 2 * p.Ncols <= kTmemCols ? 2 : 1;
  p.idesc0 = idesc_bf16_f32(2 * kTileV, p.n0w);
  p.idesc1 = idesc_bf16_f32(2 * kTileV, p.n1w ? p.n1w : 16);
  const int fixed = pair_layout(p.Ncols, 0).total;
  p.stages = (kSmemMax - fixed) / pair_layout(p.Ncols, 0).stage;
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  if (p.stages < 2) return fail(SPADE_ERR_SHAPE, "shared memory too small for R = %d", c.R);

  CUtensorMap tw, th0, th1;
  const uint64_t pitch = static_cast<uint64_t>(H) * 2;
  if (!encode_tmap_bf16_sw128(&tw, w_lm, H, c.V, pitch, kKChunk, p.th) ||
      !encode_tmap_bf16_sw128(&th0, hidden, H, c.R, pitch, kKChunk, p.n0w / 2))
    return SPADE_ERR_CUDA;
  th1 = th0;
  if (p.n1w && !encode_tmap_bf16_sw128(&th1, hidden, H, c.R, pitch, kKChunk, p.n1w / 2)) return SPADE_ERR_CUDA;

  static OncePerDevice once;
  const cudaError_t es = set_max_smem(once, kSmemMax, lm_head_pairs_kernel);
  if (es != cudaSuccess) return cuda_fail(es, "cudaFuncSetAttribute(lm_head_pairs)");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c.NC);
  cfg.blockDim = dim3(kPairThreads);
  cfg.dynamicSmemBytes = pair_layout(p.Ncols, p.stages).total;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;  // CTAs 2j, 2j + 1 share a cluster
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, lm_head_pairs_kernel, p, tw, th0, th1);
  if (e != cudaSuccess) return cuda_fail(e, "lm_head_pairs launch");
  return SPADE_OK;
}

}  // namespace accept
}  // namespace spade
