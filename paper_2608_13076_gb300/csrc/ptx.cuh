// ptx.cuh -- thin inline-PTX wrappers for sm_103a: mbarrier, TMA, bulk copies,
// cluster addressing, tcgen05 (TMEM allocation, MMA, loads/stores, fences).
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_bf16.h>

#define SPADE_DEVICE __device__ __forceinline__

namespace spade {

// Bound on every device-side wait (nanoseconds of %globaltimer).  A wait that
// expires sets SPADE_DEV_TIMEOUT and the kernel runs to its end without
// waiting again, so no launch can spin forever.
constexpr uint64_t kWaitLimitNs = 2000000000ull;

SPADE_DEVICE uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

SPADE_DEVICE uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// 2^x on the SFU (ex2.approx, relative error ~2^-22; ex2(-inf) = +0).
SPADE_DEVICE float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---------------------------------------------------------------- mbarrier
SPADE_DEVICE void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
SPADE_DEVICE void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
SPADE_DEVICE void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Orders this thread's view of generic-proxy accesses (shared and global memory)
// against the async proxy's.
SPADE_DEVICE void fence_proxy_async() { asm volatile("fence.proxy.async;" ::: "memory"); }
SPADE_DEVICE void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
SPADE_DEVICE void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// How long (ns) a try_wait may keep its thread suspended in hardware.  Without
// this hint it returns at once while the phase is pending, and the waiting warps
// of a CTA (eight epilogue warps through a whole stream) poll in a loop that takes
// issue slots and shared-memory cycles from the producer and the MMA thread.
constexpr uint32_t kSuspendNs = 1000000;
SPADE_DEVICE bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs)
      : "memory");
  return ok != 0;
}

// Whether phase `parity` has completed, without suspending the thread.
SPADE_DEVICE bool mbar_test_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for phase `parity` of `bar`.  `abort` is a CTA-shared flag: once
// any wait of the CTA has expired every later wait returns at once (the flag is
// read before a wait may suspend its thread; a completed phase is seen without it.
// The test that comes first costs nothing: projection of 72 rows 13.6 -> 13.3 us,
// attention and LM head as before).  Returns false if this wait expired (the caller records the status).
SPADE_DEVICE bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort) {
  if (mbar_test_wait(bar, parity) || *abort) return true;
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  while (true) {
    if (*abort) return true;
    if (mbar_try_wait(bar, parity)) return true;
    if (globaltimer() - t0 > kWaitLimitNs) {
      *abort = 1;
      return false;
    }
  }
}

// Bounded wait that ignores the abort flag: used to drain copies already in
// flight before a CTA exits after an expired wait.
SPADE_DEVICE bool mbar_wait_unabortable(uint64_t *bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  while (!mbar_try_wait(bar, parity)) {
    if (globaltimer() - t0 > kWaitLimitNs) return false;
  }
  return true;
}

// ---------------------------------------------------------------- warp-uniform issue
// The operands of copies, MMAs and commits sit in uniform registers.  A role whose
// loop runs on one lane keeps its values in per-thread registers and moves every
// operand over for every instruction (~110 cycles per MMA, ~350 per copy, measured);
// a role whose whole warp walks the loop, with one elected lane issuing, keeps
// them uniform.
SPADE_DEVICE int uniform_warp() { return __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0); }
// The same value on every lane, in a uniform register (a warp's lanes agree on v).
SPADE_DEVICE int uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }
template <class T>
SPADE_DEVICE T *uniform(T *v) {
  return reinterpret_cast<T *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(v), 0));
}
SPADE_DEVICE bool elect_one() {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(r));
  return r != 0;
}
// Bounded wait of a whole warp (all lanes get the same answer): true once the
// phase has completed, false if this or an earlier wait of the CTA expired.
// (An earlier expiry is seen before the wait may suspend the warp.)
SPADE_DEVICE bool warp_wait(uint64_t *bar, uint32_t parity, volatile int *abort) {
  if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
  if (__any_sync(0xffffffffu, *abort != 0)) return false;
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const uint64_t t0 = globaltimer();
  bool done = false, give_up = false;
  while (!done && !give_up) {
    done = mbar_try_wait(bar, parity);
    if (!done) {
      if (globaltimer() - t0 > kWaitLimitNs) *abort = 1;
      give_up = *abort != 0;
    }
  }
  return __all_sync(0xffffffffu, done);
}

// ---------------------------------------------------------------- programmatic dependent launch
// Waits until the grids this launch depends on have completed and their
// writes are visible; a no-op for a launch without the programmatic attribute.
SPADE_DEVICE void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next grid in the stream be scheduled before this one ends; that
// grid still waits (griddep_wait) for this grid's completion before it reads
// anything this grid writes.
SPADE_DEVICE void griddep_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ---------------------------------------------------------------- TMA
SPADE_DEVICE void tma_prefetch_desc(const CUtensorMap *map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
SPADE_DEVICE uint64_t l2_policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
SPADE_DEVICE uint64_t l2_policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
// Plain bulk copy of `bytes` from global to shared memory, completing on
// `bar`.  Both addresses 16-byte aligned; `bytes` a multiple of 16.
SPADE_DEVICE void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(static_cast<uint64_t>(__cvta_generic_to_global(src))), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// 2-D tiled load of box {x: inner, y: rows} at coordinates (x, y) into smem,
// completing `bytes` on `bar`.  x * elemsize must be a multiple of 16 bytes.
SPADE_DEVICE void tma_load_2d(void *dst, const CUtensorMap *map, int32_t x, int32_t y,
                              uint64_t *bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// 3-D tiled load of box {x, y, z} at coordinates (x, y, z); see tma_load_2d.
SPADE_DEVICE void tma_load_3d(void *dst, const CUtensorMap *map, int32_t x, int32_t y, int32_t z,
                              uint64_t *bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// Bulk copy from this CTA's shared memory to another CTA's of the cluster (both
// addresses from cluster_map), completing on that CTA's mbarrier.
SPADE_DEVICE void bulk_copy_cluster(uint32_t dst_cluster, const void *src, uint32_t bytes, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_cluster),
      "r"(smem_u32(src)), "r"(bytes), "r"(bar_cluster)
      : "memory");
}

// 4-D tiled load of box {x, y, z, u}; see tma_load_2d.
SPADE_DEVICE void tma_load_4d(void *dst, const CUtensorMap *map, int32_t x, int32_t y, int32_t z, int32_t u,
                              uint64_t *bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(u), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

SPADE_DEVICE uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

// ---------------------------------------------------------------- tcgen05
// Allocation is warp-wide; the TMEM base address is written to `dst` (smem).
SPADE_DEVICE void tmem_alloc(uint32_t *dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst)),
               "r"(ncols)
               : "memory");
}
SPADE_DEVICE void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
SPADE_DEVICE void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
SPADE_DEVICE void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
SPADE_DEVICE void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
// D(tmem) = A(smem desc) * B(smem desc)^T (+ D if accumulate), kind::f16.
SPADE_DEVICE void tc_mma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive once on `bar` when every tcgen05.mma issued so far by this thread is done.
SPADE_DEVICE void tc_commit(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}
// Each thread of the warp reads 8 consecutive 32-bit columns of its own lane.
SPADE_DEVICE void tmem_ld8(uint32_t taddr, uint32_t *r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
}
SPADE_DEVICE void tmem_st8(uint32_t taddr, const uint32_t *r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}
SPADE_DEVICE void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
SPADE_DEVICE void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---- CTA pairs (a cluster of two CTAs on two SMs, tcgen05 cta_group::2) ----
// Allocation, MMA and commit for a pair: both CTAs allocate collectively (the
// same columns in both SMs' TMEM); one thread of the even CTA issues the MMA
// with M = 256 (A rows 0-127 from its own shared memory, 128-255 from the odd
// CTA's at the same offsets) and N split between the CTAs (each holds N / 2 B
// rows at the descriptor's offset); each CTA's TMEM receives its 128 rows.
SPADE_DEVICE uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Every thread of both CTAs (no CTA may skip it).
SPADE_DEVICE void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of the same shared-memory offset in CTA `rank` of the cluster.
SPADE_DEVICE uint32_t cluster_map(const void *p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}
SPADE_DEVICE void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr)
               : "memory");
}
// Bounded wait (as mbar_wait) with cluster-scope acquire: for barriers that
// the other CTA of the pair arrives on.
SPADE_DEVICE bool mbar_try_wait_cluster(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendNs)
      : "memory");
  return ok != 0;
}
SPADE_DEVICE bool mbar_test_wait_cluster(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
SPADE_DEVICE bool mbar_wait_cluster(uint64_t *bar, uint32_t parity, volatile int *abort) {
  if (mbar_test_wait_cluster(bar, parity) || *abort) return true;
  if (mbar_try_wait_cluster(bar, parity)) return true;  // no timer read on the fast path
  const uint64_t t0 = globaltimer();
  while (true) {
    if (*abort) return true;
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if (globaltimer() - t0 > kWaitLimitNs) {
      *abort = 1;
      return false;
    }
  }
}
// 2-D tiled load into this CTA's shared memory whose completion is signalled
// on an mbarrier of either CTA of the pair (cluster address, e.g. from
// cluster_map); x * elemsize a multiple of 16 bytes.
SPADE_DEVICE void tma_load_2d_pair(void *dst, const CUtensorMap *map, int32_t x, int32_t y,
                                   uint32_t bar_cluster_addr, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      ".L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar_cluster_addr), "l"(policy)
      : "memory");
}
SPADE_DEVICE void tmem_alloc_pair(uint32_t *dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst)),
               "r"(ncols)
               : "memory");
}
SPADE_DEVICE void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
SPADE_DEVICE void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
SPADE_DEVICE void tc_mma_f16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                  uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive once on `bar` in both CTAs of the pair when every pair MMA issued so
// far by this thread is done.
SPADE_DEVICE void tc_commit_pair(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
      "[%0], %1;" ::"r"(smem_u32(bar)),
      "h"(static_cast<uint16_t>(3))
      : "memory");
}

// Shared-memory matrix descriptor for tcgen05.mma: K-major operand stored as
// 128-byte rows with the 128B swizzle (what TMA writes with
// CU_TENSOR_MAP_SWIZZLE_128B and a 64-element bf16 inner box), 8-row groups
// 1024 bytes apart.  Advancing K by 16 elements adds 32 bytes to the start.
SPADE_DEVICE uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFF) >> 4);        // start address
  d |= static_cast<uint64_t>(1) << 16;                        // leading byte offset (unused)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;                // stride byte offset
  d |= static_cast<uint64_t>(1) << 46;                        // descriptor version (sm_100)
  d |= static_cast<uint64_t>(2) << 61;                        // swizzle: 128B
  return d;
}
// Instruction descriptor of kind::f16 with bf16 A/B, fp32 D, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(uint32_t M, uint32_t N) {
  return (1u << 4)            // D format fp32
         | (1u << 7)          // A format bf16
         | (1u << 10)         // B format bf16
         | ((N >> 3) << 17)   // N / 8
         | ((M >> 4) << 24);  // M / 16
}

}  // namespace spade
