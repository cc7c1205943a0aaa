// tcgen05 / mbarrier PTX wrappers and shared-memory operand layout helpers used by the
// tensor-core weight-gradient kernels (sm_100a).
#pragma once

#include "surgeon_internal.cuh"

namespace surgeon {
namespace tc {

constexpr uint32_t kWaitCap = 1u << 22;

// ---- PTX wrappers ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait; false when it gave up.  `sleep_ns` > 0 backs off between polls (long waits).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t sleep_ns = 0) {
  for (uint32_t i = 0; i < kWaitCap; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (sleep_ns) __nanosleep(sleep_ns);
  }
  return false;
}
// The same wait, letting the hardware suspend the thread for up to about a microsecond per try
// (it wakes when the phase completes), so that a waiting thread issues almost nothing.  Bounded.
__device__ __forceinline__ bool mbar_wait_suspend(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < (1u << 21); ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(1000u)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
// TMA: 3-D tiled load global -> shared, completion counted in bytes on an mbarrier.
__device__ __forceinline__ void tma_load_3d(uint32_t smem_dst, const void* tmap, int x, int y,
                                            int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_dst), "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
// Bulk (untiled) copy global -> shared, completion counted in bytes on an mbarrier.  Both
// addresses 16-byte aligned, `bytes` a multiple of 16.
__device__ __forceinline__ void bulk_load(uint32_t smem_dst, const void* gsrc, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(smem_dst), "l"(gsrc), "r"(bytes), "r"(bar)
      : "memory");
}
// TMA: 2-D tiled load global -> shared, completion counted in bytes on an mbarrier.
__device__ __forceinline__ void tma_load_2d(uint32_t smem_dst, const void* tmap, int x, int y,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_dst), "l"(tmap), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_prefetch_desc(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t smem_dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b,
                                          uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the mbarrier once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 16 accumulator columns of a warp's 32 TMEM lanes (r: this lane's) into 16 rows of a row-major fp32 array whose
// columns are the lanes: element (e, lane) at dst[e * pitch + lane], for e < n_rows and lane < n_lanes.  `buf`: 2 KB
// of the warp's own in shared memory.  Through it the warp stores 16 bytes per lane where the rows are
// 16-byte aligned (`vec`): 16 stores of 4 bytes per lane took 1500 clocks a block, 8 us for the 512 columns of
// a CTA, as long as a small layer's products.  `at`: index of dst in an array of `limit` elements.
__device__ __forceinline__ void store_cols16(float* buf, const uint32_t (&r)[16], float* dst, long long pitch,
                                             int n_rows, int n_lanes, bool vec, long long at, long long limit,
                                             uint32_t* status) {
  const int lane = static_cast<int>(lane_id());
  if (vec) {
    __syncwarp();                                // the previous block has been read out
#pragma unroll
    for (int e = 0; e < 16; ++e) buf[e * 32 + lane] = __uint_as_float(r[e]);
    __syncwarp();
    const int c = 4 * (lane & 7);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int e = 4 * i + (lane >> 3);
      const float4 v = *reinterpret_cast<const float4*>(buf + e * 32 + c);
      if (e < n_rows && c < n_lanes && SURGEON_IN_BOUNDS(at + e * pitch + c + 3, limit, status))
        *reinterpret_cast<float4*>(dst + e * pitch + c) = v;
    }
  } else if (lane < n_lanes) {
#pragma unroll
    for (int e = 0; e < 16; ++e)
      if (e < n_rows && SURGEON_IN_BOUNDS(at + e * pitch + lane, limit, status)) dst[e * pitch + lane] = __uint_as_float(r[e]);
  }
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of 128 bytes, groups
// of 8 rows 1024 bytes apart (tile base 1024-byte aligned).
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);  // start address, 16-byte units
  d |= static_cast<uint64_t>(1) << 16;                  // leading byte offset (unused with swizzle)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;          // stride byte offset between 8-row groups
  d |= static_cast<uint64_t>(1) << 46;                  // descriptor version of this architecture
  d |= static_cast<uint64_t>(2) << 61;                  // 128-byte swizzle
  return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M x N tile.
__host__ __device__ inline uint32_t make_idesc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(m >> 4) << 24);
}

// Byte offset of 16-byte chunk `chunk` (0..7) of row `row` inside a swizzled K-major tile.
__device__ __forceinline__ uint32_t tile_off(int row, int chunk) {
  return static_cast<uint32_t>(row) * 128u + (static_cast<uint32_t>(chunk ^ (row & 7)) << 4);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
__device__ __forceinline__ unsigned short to_bf16_bits(float v) {
  return static_cast<unsigned short>(pack_bf16x2(v, 0.0f) & 0xFFFFu);
}


// ---- CTA pairs (cta_group::2): two CTAs of a cluster of 2 act as one MMA of M = 256 ---------
// Each CTA holds 128 rows of A, half of the N rows of B and its own 128 x N accumulator; the
// CTA of rank 0 issues the MMAs and owns the "full" barriers, commits arrive in both CTAs.
constexpr uint32_t kPeerBitMask = 0xFEFFFFFFu;   // shared::cluster address -> the same offset in rank 0

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t smem_dst, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst),
               "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t tmem_d, uint64_t desc_a, uint64_t desc_b,
                                               uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(desc_a), "l"(desc_b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the mbarrier at this offset in both CTAs of the pair once the MMAs issued so far
// have completed.
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(bar), "h"(static_cast<unsigned short>(3))
      : "memory");
}
// TMA load into this CTA's shared memory whose bytes count on rank 0's mbarrier at offset `bar`.
__device__ __forceinline__ void tma_load_3d_pair(uint32_t smem_dst, const void* tmap, int x, int y,
                                                 int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_dst), "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(bar & kPeerBitMask)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t smem_dst, const void* tmap, int x, int y,
                                                 uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_dst), "l"(tmap), "r"(x), "r"(y), "r"(bar & kPeerBitMask)
      : "memory");
}
// Arrive (release at cluster scope) on rank 0's mbarrier at offset `bar`.
__device__ __forceinline__ void mbar_arrive_rank0(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar & kPeerBitMask)
               : "memory");
}
// Suspended bounded wait with acquire at cluster scope (data written by the other CTA).
__device__ __forceinline__ bool mbar_wait_suspend_cluster(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < (1u << 21); ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(1000u)
        : "memory");
    if (ok) return true;
  }
  return false;
}
__device__ __forceinline__ void fence_proxy_async_all() {
  asm volatile("fence.proxy.async;" ::: "memory");
}

// The MMAs of one K-tile of 64: four K-steps into each of N_ACC accumulators of `acc_n` columns.
// `da` / `db` are the descriptors of the stage's operands; a K-step advances the start-address
// field by KSTEP (16-byte units: 2 for K-major rows, 128 for MN-major slabs), an accumulator's B
// rows lie `acc_inc` units further.  The issuing thread's own instructions are the bound of
// the tensor pipe when they are many (each MMA of 128 columns lasts only 64 clocks), so
// nothing here is computed per MMA beyond two additions.
template <int N_ACC, int KSTEP, int PAIR = 0>
__device__ __forceinline__ void umma_ktile(uint32_t tmem_base, uint32_t acc_n, uint64_t da, uint64_t db,
                                           uint64_t acc_inc, uint32_t idesc, uint32_t accum) {
#pragma unroll
  for (int a = 0; a < N_ACC; ++a) {
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      if (PAIR)
        umma_bf16_pair(tmem_base + a * acc_n, da + static_cast<uint64_t>(kk * KSTEP),
                       db + a * acc_inc + static_cast<uint64_t>(kk * KSTEP), idesc, kk > 0 ? 1u : accum);
      else
        umma_bf16(tmem_base + a * acc_n, da + static_cast<uint64_t>(kk * KSTEP),
                  db + a * acc_inc + static_cast<uint64_t>(kk * KSTEP), idesc, kk > 0 ? 1u : accum);
    }
  }
}

// Predicated load of packed value `idx` (zero when !on); no branch.
template <int DT>
__device__ __forceinline__ uint32_t ld_packed(const void* __restrict__ values, uint32_t idx, bool on) {
  uint32_t r = 0;
  const unsigned char* src =
      reinterpret_cast<const unsigned char*>(values) + static_cast<size_t>(idx) * (DT == 0 ? 4 : 2);
  if (DT == 0)
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.u32 %0, [%1];\n\t}"
                 : "+r"(r) : "l"(src), "r"(static_cast<uint32_t>(on)));
  else
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.u16 %0, [%1];\n\t}"
                 : "+r"(r) : "l"(src), "r"(static_cast<uint32_t>(on)));
  return r;
}

}  // namespace tc
}  // namespace surgeon
