// qkv_cluster.cu -- the verify block's QKV projection with rotary embedding
// (the attention input side of f_l in x_{l+1} = x_l + f_l(x_l), Sec. III-A, for
// the d+1 positions of the single forward pass, Sec. III-B): few verify rows,
// where streaming W bounds it, and larger batches over wide layers.
//
// Design (GB300):
//  * Clusters of two CTAs (76 of them cover every SM; clusters of three or more
//    leave 8 to 16 SMs idle).  A cluster owns a contiguous range of the output's
//    rotary pairs, cut in quads (4 pairs: 8 rows of W, one swizzle atom), so the
//    ranges are equal whatever the head count; each of its CTAs takes half of K.
//    An SM then receives its share of W and half of x, the two partial sums meet
//    through distributed shared memory, and nothing goes through a workspace:
//    no partials in L2 (8 MB written and read at 72 rows x 4096), no waiting on
//    other clusters, so the launch need not be cooperative (that attribute costs
//    2.7 us between dependent launches).
//  * tcgen05.mma kind::f16 (bf16 in, fp32 in tensor memory) with the cluster's W
//    rows on the MMA M side and the verify rows on N.  W is seen as
//    [head][half][pair][k], so one box brings a head's piece of the range, both
//    halves of its pairs; a range is one to three pieces, packed back to back.
//    Each piece is one box of its exact size (a tensor map per size in use):
//    copies cost ~50 ns each to issue, and pieces cut into boxes of 32, 8 and 4
//    pairs streamed at 58 GB/s per SM (25.6 us for the Llama-3-8B layer).  The
//    last 128-row operand of a stage may read past its valid rows (into the
//    stage's x rows or the next stage: lanes that are never read); the ring is
//    followed by at least 16 KB of staging so that this stays in plain buffers.
//  * A ring slot's round trip (MMAs done, slot released, copies issued, data
//    landed, MMA thread woken) is ~2.2 us whether W comes from HBM or L2, so the
//    stream's rate is the bytes in flight: one-chunk stages packed without
//    padding, as many as fit (8 of 21 KB at the Llama-3-8B layer).
//  * Epilogue: accumulators go to shared memory; the columns of the verify rows
//    that the peer finishes travel there by one bulk copy (scalar remote stores
//    took 4.6 us), and each CTA sums, rotates and stores its half of the rows.
//    With many rows the staging takes the ring's place once both CTAs' MMAs are
//    done, as many verify rows at a time as fit.
#include "qkv_common.cuh"

namespace spade {
namespace qkv {
namespace pair {

constexpr int kThreads = 320;                  // producer warp, MMA warp, eight epilogue warps
constexpr int kEpiThreads = 256;
constexpr int kMaxRows = 512;                  // verify rows
constexpr int kMaxStages = 12;
constexpr int kMinStages = 4;                  // staging beside the ring
constexpr int kMinStagesOver = 3;              // staging in the ring's place
constexpr int kBatch = 128;                    // verify rows that the ring's place must take at once
constexpr int kMaxPiece = 16;                  // quads of a piece (a head of dimension 128)
constexpr int kMaxQuads = 64;                  // quads of a cluster's range (512 rows)
constexpr int kSmemBudget = 222 * 1024;
constexpr int kTileBytes = 128 * kKChunk * 2;  // one 128-row operand x one k-chunk

struct Maps {
  CUtensorMap w[kMaxPiece];  // boxes of 1 .. 16 quads (those in use)
  CUtensorMap x0, x1;        // verify rows up to 256, the rest
};

struct Params {
  Call c;
  int quads, nclusters;  // quads of the output, clusters
  int qmax;              // most quads of a cluster
  int KC;                // k-chunks (ceil(H / 64))
  int Ncols;             // verify rows rounded up to 16: MMA N
  int stages;
  int over;              // staging in the ring's place
  int batch;             // verify rows staged at once (R when the staging has its own room)
  uint32_t tmem_cols;
};

// Shared-memory plan (offsets from a 1024-byte aligned base): tables first, then
// the ring, then the staging (or, in the ring's place, a pad for the last
// operand's read): this CTA's partial sums of a batch of verify rows, and those
// received for the rows that it finishes.
struct Layout {
  int rseq, rpos, freq, qrow, bars, misc, ring, stage_bytes, row_stride, part, recv, region, total;
};
__host__ __device__ inline Layout layout(int Ncols, int qmax, int stages, int over, int batch) {
  Layout L;
  L.rseq = 0;
  L.rpos = L.rseq + kMaxRows * 4;
  L.freq = L.rpos + kMaxRows * 4;
  L.qrow = L.freq + 64 * 4;  // uint16 [kMaxQuads][2]
  L.bars = L.qrow + kMaxQuads * 4;
  L.misc = L.bars + (2 * kMaxStages + 3) * 8;
  L.ring = (L.misc + 32 + 1023) & ~1023;
  L.stage_bytes = qmax * 1024 + Ncols * 128;  // 8 W rows per quad, then the x rows
  const int end = L.ring + stages * L.stage_bytes;
  L.row_stride = qmax * 8 + 4;                // floats per staged verify row
  const int staging = (batch + (batch + 1) / 2) * L.row_stride * 4;  // (a multiple of 16)
  L.part = over ? L.ring : end;
  L.recv = L.part + batch * L.row_stride * 4;
  L.region = staging;  // the next batch's (in the ring's place)
  L.total = end + (over || staging < kTileBytes ? kTileBytes : staging) + 1024;  // + slack for the 1024-byte alignment
  return L;
}

__device__ __forceinline__ void epi_bar() {
  __syncwarp();
  asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
}

// kBig: more than 128 verify rows are possible (a second N-chunk, staging in the
// ring's place); the small form has neither test in its loops.
template <bool kBig>
__global__ void __launch_bounds__(kThreads, 1)
    qkv_cluster_kernel(const __grid_constant__ Params p, const __grid_constant__ Maps maps) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const Layout L = layout(p.Ncols, p.qmax, p.stages, p.over, p.batch);
  uint32_t *s_row = reinterpret_cast<uint32_t *>(smem + L.rseq);
  int32_t *s_rpos = reinterpret_cast<int32_t *>(smem + L.rpos);
  float *s_freq = reinterpret_cast<float *>(smem + L.freq);
  uint16_t *s_qrow = reinterpret_cast<uint16_t *>(smem + L.qrow);
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + L.bars);
  uint64_t *empty = full + kMaxStages;
  uint64_t *acc_full = empty + kMaxStages;
  uint64_t *recv_full = acc_full + 1;  // [2]: the peer's partial sums of a batch have landed
  uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + L.misc);
  volatile int *s_abort = reinterpret_cast<volatile int *>(smem + L.misc + 8);

  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  const int cl = blockIdx.x >> 1;
  const int q0 = static_cast<int>(static_cast<int64_t>(p.quads) * cl / p.nclusters);
  const int nq = static_cast<int>(static_cast<int64_t>(p.quads) * (cl + 1) / p.nclusters) - q0;
  const int rows = nq * 8;                  // W rows of the cluster
  const int ntile = (rows + 127) / 128;     // 128-row operands
  const int qph = p.c.D / 8;                // quads per head
  const int n0 = kBig ? min(p.Ncols, 256) : p.Ncols, n1 = kBig ? p.Ncols - n0 : 0;  // MMA N-chunks
  // Of the nb verify rows of a batch, the first half is finished by CTA 0.
  auto own_rows = [rank](int nb) { return rank ? nb - (nb + 1) / 2 : (nb + 1) / 2; };
  // Arms the barrier of batch i (if there is one) with the bytes that the peer sends.
  const int nbatch = kBig ? (p.c.R + p.batch - 1) / p.batch : 1;
  auto arm = [&](int i) {
    if (i < nbatch)
      mbar_arrive_expect_tx(&recv_full[i & 1],
                            static_cast<uint32_t>(own_rows(min(p.batch, p.c.R - i * p.batch)) * L.row_stride * 4));
  };
  // This CTA's half of K.  Every cluster reads the same x rows: each starts at
  // another chunk, so that they do not all load the same lines from L2 at once.
  const int kc0 = p.KC * static_cast<int>(rank) / 2, nk = p.KC * (static_cast<int>(rank) + 1) / 2 - kc0;
  const int rot = nk > 0 ? cl % nk : 0;

  // ---- set-up that reads no input -----------------------------------------
  if (tid == 0) *s_abort = 0;
  for (int j = tid; j < p.c.D / 2; j += kThreads) s_freq[j] = p.c.inv_freq[j];
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&maps.x0);
    if (n1) tma_prefetch_desc(&maps.x1);
    // Pieces: one box per head.  A box lands as its pairs' rows of the first
    // half, then of the second; s_qrow: where a quad's four rows of each half start.
    for (int q = q0; q < q0 + nq;) {
      const int j = q % qph, take = min(qph - j, q0 + nq - q);
      tma_prefetch_desc(&maps.w[take - 1]);
      for (int i = 0; i < take; ++i) {
        s_qrow[2 * (q - q0 + i)] = static_cast<uint16_t>((q - q0) * 8 + i * 4);
        s_qrow[2 * (q - q0 + i) + 1] = static_cast<uint16_t>((q - q0) * 8 + (take + i) * 4);
      }
      q += take;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      for (int s = 0; s < p.stages; ++s) {
        mbar_init(&full[s], 1);
        mbar_init(&empty[s], 1);
      }
      mbar_init(acc_full, 1);
      mbar_init(&recv_full[0], 1);
      mbar_init(&recv_full[1], 1);
      fence_mbar_init();
      arm(0);
      if (kBig) arm(1);
    }
    __syncwarp();
    tmem_alloc(s_tmem, p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the peer runs: its shared memory may be written from here on
  tc_fence_after();
  // Inputs written by earlier kernels in the stream are visible from here on.
  griddep_wait();
  griddep_launch_dependents();
  const uint32_t tmem = *s_tmem;
  const int xoff = p.qmax * 1024;

  if (warp == 0) {
    // ============================ producer: TMA ============================
    const bool leader = elect_one();
    const uint64_t pol_w = l2_policy_evict_first();  // W streams once
    const uint64_t pol_x = l2_policy_evict_last();   // x is re-read by every cluster
    const uint32_t bytes = static_cast<uint32_t>(rows * 128 + p.Ncols * 128);
    const int h_first = q0 / qph, j_first = q0 - h_first * qph;
    int s = 0, issued = 0, kc = kc0 + rot;
    uint32_t ph = 1;
    bool ok = true;
    for (; issued < nk; ++issued) {
      ok = warp_wait(&empty[s], ph, s_abort);
      if (!ok) break;
      uint8_t *stage = smem + L.ring + s * L.stage_bytes;
      const int kx = kc * kKChunk;
      if (leader) mbar_arrive_expect_tx(&full[s], bytes);
      // The range's pieces, one box per head.
      for (int q = 0, h = h_first, j = j_first; q < nq; ++h, j = 0) {
        const int take = min(qph - j, nq - q);
        if (leader) tma_load_4d(stage + q * 1024, &maps.w[take - 1], kx, j * 4, 0, h, &full[s], pol_w);
        q += take;
      }
      if (leader) tma_load_2d(stage + xoff, &maps.x0, kx, 0, &full[s], pol_x);
      if (n1) {
        if (leader) tma_load_2d(stage + xoff + n0 * 128, &maps.x1, kx, n0, &full[s], pol_x);
      }
      if (++kc == kc0 + nk) kc = kc0;
      if (++s == p.stages) { s = 0; ph ^= 1u; }
    }
    if (!ok && leader) {
      atomicOr(p.c.status, SPADE_DEV_TIMEOUT);
      // Drain: every copy issued must land before shared memory goes away.
      for (int i = (issued > p.stages ? issued - p.stages : 0); i < issued; ++i)
        mbar_wait_unabortable(&full[i % p.stages], (i / p.stages) & 1);
    }
  } else if (warp == 1) {
    // ============================ MMA issuer ===============================
    const bool leader = elect_one();
    const uint32_t idesc0 = idesc_bf16_f32(128, n0), idesc1 = idesc_bf16_f32(128, n1 ? n1 : 16);
    int s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int it = 0; it < nk; ++it) {
      ok = warp_wait(&full[s], ph, s_abort);
      if (!ok) break;  // (an expired wait of the CTA: the results are void)
      tc_fence_after();
      const uint32_t base = smem_u32(smem + L.ring + s * L.stage_bytes);
      // Descriptors built once per operand; a K step of 16 adds 32 bytes, 2 in
      // the descriptor's address field.
      const uint64_t db0 = smem_desc_sw128(base + xoff), db1 = smem_desc_sw128(base + xoff + n0 * 128);
      for (int t = 0; t < ntile; ++t) {
        const uint64_t da = smem_desc_sw128(base + t * kTileBytes);
        const uint32_t d = tmem + static_cast<uint32_t>(t * p.Ncols);
#pragma unroll
        for (int kk = 0; kk < kKChunk / 16; ++kk) {
          if (leader) tc_mma_f16(d, da + 2u * kk, db0 + 2u * kk, idesc0, (it > 0 || kk > 0) ? 1u : 0u);
          if (n1) {
            if (leader) tc_mma_f16(d + 256u, da + 2u * kk, db1 + 2u * kk, idesc1, (it > 0 || kk > 0) ? 1u : 0u);
          }
        }
      }
      if (leader) tc_commit(&empty[s]);
      if (++s == p.stages) { s = 0; ph ^= 1u; }
    }
    if (nk > 0 && leader) {
      tc_commit(acc_full);
      if (!ok) {
        atomicOr(p.c.status, SPADE_DEV_TIMEOUT);
        // Every MMA issued must be done before its operands and the tensor memory go away.
        mbar_wait_unabortable(acc_full, 0);
      }
    }
  } else {
    // ===================== epilogue warps: wait for the accumulators =======
    build_rows(p.c, s_row, s_rpos, tid - 64, kEpiThreads, [] { epi_bar(); });
    if (nk > 0) {
      if (!mbar_wait(acc_full, 0, s_abort)) atomicOr(p.c.status, SPADE_DEV_TIMEOUT);
      tc_fence_after();
    }
  }
  if constexpr (kBig) {
    __syncwarp();
    __syncthreads();
    cluster_sync();  // both rings are idle: their place becomes staging
  }
  const OutMap om = out_map(p.c);
  // Batches alternate between two regions: this CTA's sums of the batch's rows, then
  // those received from the peer for the rows that this CTA finishes.
  auto part_of = [&](int i) { return reinterpret_cast<float *>(smem + L.part + (kBig ? i & 1 : 0) * L.region); };
  auto recv_of = [&](int i) { return reinterpret_cast<float *>(smem + L.recv + (kBig ? i & 1 : 0) * L.region); };
  // Batch i from tensor memory to its region, and the peer's rows on their way
  // (epilogue warps).
  auto stage = [&](int i) {
    const int b0 = i * p.batch, nb = kBig ? min(p.batch, p.c.R - b0) : p.c.R;
    const int n_own = own_rows(nb), n_send = nb - n_own, first_send = rank ? 0 : n_own;
    float *part = part_of(i);
    // Two warps per lane quarter, each every second 16 columns.
    const int q4 = warp & 3;
    for (int t = 0; t < ntile; ++t) {
      if (t * 128 + q4 * 32 >= rows) break;  // (whole warps: rows is a multiple of 8)
      const int row = t * 128 + q4 * 32 + lane;
      const uint32_t a = tmem + (static_cast<uint32_t>(q4 * 32) << 16) + static_cast<uint32_t>(t * p.Ncols + b0);
      for (int c = 16 * ((warp - 2) >> 2); c < nb; c += 32) {
        uint32_t v[16];
        if (nk > 0) {
          tmem_ld8(a + c, v);
          tmem_ld8(a + c + 8, v + 8);
          tmem_wait_ld();
        } else {  // (one k-chunk in all: this CTA has none)
#pragma unroll
          for (int e = 0; e < 16; ++e) v[e] = 0u;
        }
        if (row < rows) {
          float *to = part + c * L.row_stride + row;
#pragma unroll
          for (int e = 0; e < 16; ++e)
            if (c + e < nb) to[e * L.row_stride] = __uint_as_float(v[e]);
        }
      }
    }
    // The peer's rows travel in one copy.
    fence_proxy_async_smem();
    epi_bar();
    if (tid == 64 && n_send > 0)
      bulk_copy_cluster(cluster_map(recv_of(i), rank ^ 1u), part + first_send * L.row_stride,
                        static_cast<uint32_t>(n_send * L.row_stride * 4), cluster_map(&recv_full[kBig ? i & 1 : 0], rank ^ 1u));
  };
  const int dn = kThreads / nq, dq = kThreads - dn * nq, qsh = p.c.D == 128 ? 4 : 3;
  if (warp >= 2) {
    stage(0);
    if (kBig && nbatch > 1) stage(1);
  }
#pragma unroll 1
  for (int i = 0; i < nbatch; ++i) {
    const int b0 = i * p.batch, nb = kBig ? min(p.batch, p.c.R - b0) : p.c.R, n_own = own_rows(nb);
    const int first = rank ? nb - n_own : 0;  // within the batch
    const float *part = part_of(i), *recv = recv_of(i);
    __syncwarp();
    __syncthreads();  // staged
    if (!mbar_wait_unabortable(&recv_full[kBig ? i & 1 : 0], kBig ? (i >> 1) & 1 : 0)) atomicOr(p.c.status, SPADE_DEV_TIMEOUT);
    // Items (verify row, quad), kThreads apart.
    for (int n = tid / nq, q = tid - n * nq; n < n_own;) {
      const int r = b0 + first + n;
      const uint32_t row = s_row[r];
      if (row != kNoRow) {
        const float *o = part + (first + n) * L.row_stride, *in = recv + n * L.row_stride;
        const int r1 = s_qrow[2 * q], r2 = s_qrow[2 * q + 1];
        const float4 o1 = *reinterpret_cast<const float4 *>(o + r1), o2 = *reinterpret_cast<const float4 *>(o + r2);
        const float4 i1 = *reinterpret_cast<const float4 *>(in + r1), i2 = *reinterpret_cast<const float4 *>(in + r2);
        float y1[4] = {o1.x + i1.x, o1.y + i1.y, o1.z + i1.z, o1.w + i1.w};
        float y2[4] = {o2.x + i2.x, o2.y + i2.y, o2.z + i2.z, o2.w + i2.w};
        const int Q = q0 + q, hg = Q >> qsh;
        store_quad(om, s_freq, row, r, s_rpos[r], hg, (Q - (hg << qsh)) * 4, y1, y2);
      }
      n += dn;
      q += dq;
      if (q >= nq) { q -= nq; ++n; }
    }
    if (kBig && i + 2 < nbatch) {
      __syncwarp();
      __syncthreads();
      // Every thread of this CTA has seen batch i's phase complete, and the peer sends
      // only after the cluster's barrier.  (A last batch of one row brings CTA 1
      // nothing: armed with 0 bytes its phase completes at once, and a thread still
      // waiting for batch i's would miss both.)
      if (tid == 0) arm(i + 2);
      __syncwarp();
      cluster_sync();  // both CTAs have read this region, and their copies have left it
      if (warp >= 2) stage(i + 2);
    }
  }
  tc_fence_before();
  __syncwarp();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, p.tmem_cols);
  }
  cluster_sync();  // the last copy to the peer has left this CTA's shared memory
}

// W [(Hq + 2 Hkv) D, H] as {H, D / 2 pairs, 2 halves, heads}, box {64, pairs, 2, 1},
// 128-byte swizzle.
static bool encode_w(CUtensorMap *map, const void *w, const Call &c, uint32_t pairs) {
  const uint64_t H = c.H, row = H * 2;
  const uint64_t dims[4] = {H, static_cast<uint64_t>(c.D / 2), 2, static_cast<uint64_t>(c.Hq + 2 * c.Hkv)};
  const uint64_t strides[3] = {row, row * (c.D / 2), row * c.D};
  const uint32_t box[4] = {kKChunk, pairs, 2, 1};
  return encode_tmap_bf16_sw128_nd(map, w, 4, dims, strides, box);
}

// Plan for these sizes; stages = 0 when the form does not take them.
static Params plan(const Call &c, int sms) {
  Params p{};
  p.c = c;
  p.quads = (c.Hq + 2 * c.Hkv) * c.D / 8;
  p.nclusters = sms / 2 < p.quads ? sms / 2 : p.quads;
  if (c.R > kMaxRows || p.nclusters < 1) return p;
  p.qmax = (p.quads + p.nclusters - 1) / p.nclusters;
  p.KC = (c.H + kKChunk - 1) / kKChunk;
  p.Ncols = (c.R + 15) / 16 * 16;
  const int cols = (p.qmax * 8 + 127) / 128 * p.Ncols;  // accumulator columns
  if (cols > 512 || p.qmax > kMaxQuads) return p;
  p.tmem_cols = 32;
  while (p.tmem_cols < static_cast<uint32_t>(cols)) p.tmem_cols *= 2;
  auto depth = [&](int over, int batch) {
    const Layout L = layout(p.Ncols, p.qmax, 0, over, batch);
    const int n = (kSmemBudget - L.total) / L.stage_bytes;
    return n > kMaxStages ? kMaxStages : n;
  };
  int n = depth(0, c.R);
  if (c.R <= 128 && n >= kMinStages) {
    p.stages = n;
    p.batch = c.R;
    return p;
  }
  // More rows: every cluster reads all of x, so its range must have enough W rows
  // (64) for the x rows it loads; the stream-K form has 128 per x row.
  n = depth(1, kBatch);
  const Layout L = layout(p.Ncols, p.qmax, n, 1, kBatch);
  if (p.qmax >= 8 && n >= kMinStagesOver && L.recv + kBatch / 2 * L.row_stride * 4 <= L.ring + n * L.stage_bytes) {
    p.stages = n;
    p.over = 1;
    // Two regions, so that a batch's exchange and staging run under the one before
    // it; at least two batches, as few as fit, of nearly equal sizes (multiples of 16).
    // 389 paged rows x 5120 x 7168: 33.7 us; in one region 34.8 (two batches) and
    // 40.7 (four, with pages looked up and divisions per item).
    const int fit = n * L.stage_bytes / (L.row_stride * 12) / 16 * 16;
    const int nb = c.R > 2 * fit ? (c.R + fit - 1) / fit : 2;
    p.batch = ((c.R + nb - 1) / nb + 15) / 16 * 16;
  }
  return p;
}

}  // namespace pair

// Up to 128 rows the cluster form streams W at the rate its ring allows and is
// taken when at least four stages fit: 13.3 us at 72 rows against 20.5 us of the
// stream-K form. Above, see plan() (464 rows are the most whose ring fits, over ranges
// of eight quads).
bool cluster_fits(const Call &c, int sms) { return pair::plan(c, sms).stages > 0; }

spade_status launch_cluster(const Call &c, const void *x, const void *w_qkv, int sms, cudaStream_t stream) {
  using namespace pair;
  const Params p = plan(c, sms);
  Maps m;
  const uint64_t pitch = static_cast<uint64_t>(c.H) * 2;
  const int n0 = p.Ncols < 256 ? p.Ncols : 256;
  if (!encode_tmap_bf16_sw128(&m.x0, x, c.H, c.R, pitch, kKChunk, n0)) return SPADE_ERR_CUDA;
  if (p.Ncols > n0 && !encode_tmap_bf16_sw128(&m.x1, x, c.H, c.R, pitch, kKChunk, p.Ncols - n0)) return SPADE_ERR_CUDA;
  // The piece sizes that some cluster's range has.
  const int qph = c.D / 8;
  uint32_t used = 0;
  for (int cl = 0, q = 0; cl < p.nclusters; ++cl) {
    const int end = static_cast<int>(static_cast<int64_t>(p.quads) * (cl + 1) / p.nclusters);
    while (q < end) {
      const int left = qph - q % qph, take = left < end - q ? left : end - q;
      if (!(used >> (take - 1) & 1u) && !encode_w(&m.w[take - 1], w_qkv, c, 4 * take)) return SPADE_ERR_CUDA;
      used |= 1u << (take - 1);
      q += take;
    }
  }
  static OncePerDevice once;
  const cudaError_t es = set_max_smem(once, kSmemBudget, qkv_cluster_kernel<false>, qkv_cluster_kernel<true>);
  if (es != cudaSuccess) return cuda_fail(es, "cudaFuncSetAttribute(qkv_cluster)");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * p.nclusters);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = layout(p.Ncols, p.qmax, p.stages, p.over, p.batch).total;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, p.over ? qkv_cluster_kernel<true> : qkv_cluster_kernel<false>, p, m);
  if (e != cudaSuccess) return cuda_fail(e, "qkv_cluster launch");
  return SPADE_OK;
}

}  // namespace qkv
}  // namespace spade
