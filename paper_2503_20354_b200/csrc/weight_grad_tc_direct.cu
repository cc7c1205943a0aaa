// Tensor-core weight gradient for layers whose im2col operand is the activation itself: linear
// layers ([T, C] activations), 1x1 / pad 0 convolutions of stride 1 or 2, and k x k stride-1
// convolutions through shifted copies of the output gradient (NCHW).  Algorithm 1,
// Reshape and gradient steps with Eq. 2:  D[c, o] = sum_k A[k, c] * G[k, o].
//
//   c (input channel)  -> MMA M, 128 per CTA (TMEM lanes)
//   o (output channel, per tap for a k x k convolution) -> MMA N, one to three accumulators of
//                         up to 256 columns, at most 512 in all
//   k (row t, or image b and position p) -> MMA K, 64 per pipeline stage
//
// Operand layouts follow the memory order of the tensors, so that neither needs a transpose:
//   linear : A[t, c] and G[t, o] are contiguous along c / o -> both operands MN-major
//            (rows of 64 channels = 128 bytes, one row per k, 128-byte swizzle);
//   conv   : A[b, c, p] and G[b, o, p] are contiguous along p -> both operands K-major.
// The output gradient is converted to bf16 once by a streaming pre-pass and arrives by TMA.
//
// k x k layers on maps at most 64 wide (TG): the pre-pass writes ONE transposed copy, [image][position]
// [channel], which the kernel takes as an MN-major operand.  A column shift is then a box offset along
// x, which no 16-byte rule restricts because x is not the innermost dimension, with zero fill
// outside the map; a row shift is an offset along y.  (The K-major copies need one per column shift, or
// one per tap: 196 MB written and read back for 160 channels on 32x32 at batch 200, which L2 does not
// hold.)  A K-tile is as many whole map rows as fit 64 positions.  What a CTA loads per K-tile:
//   TG 1    a box per tap of its units;
//   TG 2    (rows a multiple of 8 wide) the three taps of one kernel column share a box that is kh - 1 rows
//           higher: a tap's row shift is a start address, in units of 8 k-rows;
//   TG 3-5  (16, 32, 64 wide, 3 x 3) the row shifts are whole K-steps: boxes without the extra rows
//           ("slabs"), of which the CTA keeps the ones before, at and behind the activation tile in the
//           ring; a tap's shift is a choice of slab and start address per MMA.  Every slab is loaded once.
// 160 channels on 32x32, batch 200: 247 -> 189 us a call; 640 channels on 8x8: 167 -> 145.
//
// 1x1 layers of stride 2 on maps at most 128 wide take that copy as well (MODE 3): a K-tile is 64 / slot_w output rows, each at
// a multiple of slot_w = 8, 16, 32 or 64 positions (the boxes are slot_w wide and bring zeros past a row's end), so that a
// lane's run is one, two or four pieces of input rows at places that are known when the kernel is compiled.  A run that
// began anywhere in a row was walked segment by segment and kept value by kept value (MODE 2, for the others), 13000 clocks a
// K-tile: 1024 -> 2048 channels on 14x14, batch 64, bf16, 70 % pruned 108 -> 54 us; 512 -> 1024 on 28x28 97 -> 67; 256 ->
// 512 on 56x56 97 -> 83, unpruned 165 -> 97.
//
// The activation operand is rebuilt from the compressed store by 16 producer warps, 8 per K-tile,
// two tiles in flight: a lane owns a run of 32 consecutive elements (64 bytes of the swizzled
// tile), finds the rank of its first kept element from the block offset and the block's bitmap
// words, and rebuilds the run as four 16-byte chunks with one predicated load per element (all
// independent; fp32 tiles that are mostly kept go through a coalesced per-warp staging copy
// instead).  The metadata of a lane's next run is fetched while the current one is rebuilt.
// One thread issues the MMAs, one the TMA loads; split-K partial tiles are reduced in a fixed
// order by the caller.  Every wait is bounded and ends in SURGEON_ERR_TIMEOUT.
#include <cuda.h>

#include <algorithm>
#include <cstddef>
#include <cstdlib>
#include <type_traits>

#include "surgeon_internal.cuh"
#include "tc_common.cuh"
#include "weight_grad_tc_conv.cuh"

namespace surgeon {

namespace {

using namespace tc;

constexpr int kTileM = 128;
constexpr int kTileK = 64;
constexpr int kGroups = 2;                       // producer groups of 8 warps, one K-tile in flight each
constexpr int kProdWarps = 8 * kGroups;
constexpr int kProdThreads = kProdWarps * 32;
constexpr int kThreads = 64 + kProdThreads;     // warp 0: MMA, warp 1: TMA, warps 2..17: producers
// CTA pairs (cta_group::2) halve the gradient traffic per MMA.  They measured slower than single
// CTAs while the activation producers are the bound (a pair waits for the slower of its two
// tiles), so they are off unless the environment variable SURGEON_DW_PAIRS is set to 1.
static bool use_pairs() {
  static const bool on = [] {
    const char* e = std::getenv("SURGEON_DW_PAIRS");
    return e && e[0] == '1';
  }();
  return on;
}
constexpr int kMaxAStages = 8;
constexpr uint32_t kFewMost = 12;                // kept elements of a 32-element run that are scattered one by one
constexpr int kMaxBStages = 8;
constexpr int kATileBytes = kTileM * kTileK * 2;              // 16 KB
// staging of packed values: per warp 16 rows of 64 + 16 bf16 (conv) or 8 rows of 128 + 16 (linear)
constexpr int kStageBytesPerWarp = 16 * (64 + 16) * 2;
constexpr int kStageBytes = kProdWarps * kStageBytesPerWarp;  // 40 KB

// Shared-memory matrix descriptor of an MN-major operand with 128-byte swizzle: rows of 64
// elements (128 bytes) per k, 8 rows per 1024-byte group (stride byte offset), the next 64
// elements along M/N one slab of 64 k-rows further (leading byte offset).
__device__ __forceinline__ uint64_t make_desc_mn(uint32_t saddr, int k_rows = kTileK) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((k_rows * 128) >> 4) << 16;   // leading byte offset: next 64-wide slab
  d |= static_cast<uint64_t>(1024 >> 4) << 32;             // stride byte offset: next 8 k-rows
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;                     // 128-byte swizzle
  return d;
}

__device__ __forceinline__ void tma_load_4d(uint32_t smem_dst, const void* tmap, int c, int x, int y, int img,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(smem_dst), "l"(tmap), "r"(c), "r"(x), "r"(y), "r"(img), "r"(bar)
      : "memory");
}
// One K-tile into N_ACC accumulators with a K-major A and an MN-major B (K-steps 2 and 128 units apart).
template <int N_ACC>
__device__ __forceinline__ void umma_ktile_tg(uint32_t tmem_base, uint32_t acc_n, uint64_t da, uint64_t db,
                                              uint64_t acc_inc, uint32_t idesc, uint32_t accum) {
#pragma unroll
  for (int a = 0; a < N_ACC; ++a)
#pragma unroll
    for (int kk = 0; kk < 4; ++kk)
      umma_bf16(tmem_base + a * acc_n, da + static_cast<uint64_t>(kk * 2), db + a * acc_inc + static_cast<uint64_t>(kk * 128),
                idesc, kk > 0 ? 1u : accum);
}

// What a lane fetches for the 32 consecutive elements ("word") it rebuilds: the kept count before
// their 128-element block, the block's bitmap words, and the bitmap word after the one the run
// starts in (the run need not start on a word boundary).
struct WordRaw {
  uint32_t base;
  uint32_t next;
  uint4 words;
  uint32_t j;          // flat index of the run's first element
  uint32_t nvalid;     // elements of the run that exist (0: nothing to do)
};

template <int DT, int MODE, int PAIR, int TG = 0>
__global__ void __launch_bounds__(kThreads, 1)
dw_direct_kernel(const uint32_t* __restrict__ bitmap, const void* __restrict__ values,
                 const uint32_t* __restrict__ offsets, const __grid_constant__ CUtensorMap grad_map,
                 float* __restrict__ partial, uint32_t* __restrict__ status, DirectParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  // Two rings: activation tiles (16 KB each, many) and gradient tiles (n_cols rows each, few).
  // The activation ring is deep because rebuilding a tile takes longer than its MMAs; the
  // gradient tiles arrive by TMA well ahead and need only be double- or triple-buffered.
  // In a CTA pair each CTA holds half of the gradient rows of every accumulator.
  constexpr int SLAB = TG >= 3 ? 1 << (TG - 3) : 0;      // map width in K-steps of 16
  const int b_stage_bytes = TG ? p.b_bytes : p.n_cols * (PAIR ? 64 : 128);
  const int acc_rows = PAIR ? p.acc_n / 2 : p.acc_n;     // gradient rows per accumulator in this CTA
  const uint32_t cta_rank = PAIR ? cluster_ctarank() : 0u;
  unsigned char* b_ring = smem + p.a_stages * kATileBytes;
  __shared__ __align__(8) unsigned long long bars[2 * kMaxAStages + 2 * kMaxBStages + 1];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile uint32_t fail;

  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const uint32_t lane = lane_id();
  const int m_tile = blockIdx.x, n_tile = blockIdx.y, split = blockIdx.z;
  const int c0 = m_tile * p.rows_per_tile;           // first input channel of the CTA's row tile
  const int rows_here = max(0, min(p.rows_per_tile, p.C - c0));   // tile rows that hold a channel
  const int o0 = n_tile * p.n_cols;                  // linear: first gradient column of the CTA
  const int u0 = n_tile * p.n_acc;                   // conv: first column unit of the CTA
  const int n_acc_here = (MODE == 0 || TG >= 2) ? p.n_acc : min(p.n_acc, p.n_units - u0);
  const int kt_begin = split * p.ktiles_per_split;
  const int kt_end = min(kt_begin + p.ktiles_per_split, p.total_ktiles);
  const int n_kt = kt_end - kt_begin;

  const uint32_t full_a = smem_u32(bars);
  const uint32_t empty_a = smem_u32(bars + kMaxAStages);
  const uint32_t full_b = smem_u32(bars + 2 * kMaxAStages);
  const uint32_t empty_b = smem_u32(bars + 2 * kMaxAStages + kMaxBStages);
  const uint32_t acc_bar = smem_u32(bars + 2 * kMaxAStages + 2 * kMaxBStages);
  if (tid == 0) {
    tma_prefetch_desc(&grad_map);
    for (int s = 0; s < p.a_stages; ++s) {
      mbar_init(full_a + 8 * s, (PAIR ? 2 : 1) * 8);   // the 8 warps (of each CTA) that rebuild a tile
      mbar_init(empty_a + 8 * s, 1);
    }
    for (int s = 0; s < p.b_stages; ++s) {
      mbar_init(full_b + 8 * s, 1);                    // the TMA thread (+ the bytes it expects)
      mbar_init(empty_b + 8 * s, 1);
    }
    mbar_init(acc_bar, 1);
    fail = 0;
    fence_barrier_init();
  }
  if (warp == 0) {
    if (PAIR) tmem_alloc_pair(smem_u32(&tmem_slot), p.tmem_cols);
    else tmem_alloc(smem_u32(&tmem_slot), p.tmem_cols);
  }
  if ((TG == 1 || TG == 2) && p.kpos < kTileK) {
    // the k-rows of a stage that no box fills meet zeros of the activation: they must be finite
    for (int v = tid; v < p.b_stages * b_stage_bytes / 16; v += kThreads)
      reinterpret_cast<uint4*>(b_ring)[v] = make_uint4(0, 0, 0, 0);
    fence_proxy_async();
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();          // both CTAs' barriers exist before either is arrived on
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  pdl_trigger();                         // the split reduction may be launched; it waits for this grid

  if (warp == 0) {
    // ================= MMA issuer (rank 0 of a pair) =================
    if (lane == 0 && cta_rank == 0) {
      const uint32_t idesc = make_idesc(PAIR ? 2 * kTileM : kTileM, p.acc_n) | (MODE == 0 ? ((1u << 15) | (1u << 16)) : (TG ? (1u << 16) : 0u));
      const uint64_t a_base = (MODE == 0) ? make_desc_mn(smem_u32(smem)) : make_desc(smem_u32(smem));
      const uint64_t b_base = (MODE == 0) ? make_desc_mn(smem_u32(b_ring))
                              : TG ? make_desc_mn(smem_u32(b_ring), p.k_rows) : make_desc(smem_u32(b_ring));
      const uint64_t a_inc = static_cast<uint64_t>(kATileBytes >> 4);
      const uint64_t b_inc = static_cast<uint64_t>(b_stage_bytes >> 4);
      // TG 1: a unit's box behind the other; TG 2: kernel row a reads the gradient a map rows before row 0's place
      const uint64_t acc_inc = TG == 1   ? static_cast<uint64_t>(p.unit_bytes >> 4)
                               : TG == 2 ? static_cast<uint64_t>(0) - static_cast<uint64_t>((p.in_w * 128) >> 4)
                                         : static_cast<uint64_t>((acc_rows * 128) >> 4);
      const uint64_t first_row = TG == 2 ? static_cast<uint64_t>(((p.kh - 1) * p.in_w * 128) >> 4) : 0u;
      constexpr int kStep = (MODE == 0) ? 128 : 2;
      uint64_t da = a_base, db = b_base;
      uint32_t pa = 0, pb = 0, accum = 0;
      int sa = 0, sb = 0;
      bool ok = true;
#ifdef SURGEON_DW_STATS
      // clock stamps of the issuing thread (a build with -DSURGEON_DW_STATS; read from the scratch
      // status area by paper_2503_20354_b200/diagnostics.py): where a K-tile's time goes
      long long st_g = 0, st_a = 0;
      const long long st_begin = clock64();
#endif
      if (SLAB) {
        // slab q of an image holds positions 64 (q - 1) ...; K-tile j needs slabs j, j + 1, j + 2
        int kin = kt_begin % p.tiles_per_img;
        int slot = 0;                              // of slab kin; the two behind it follow in the ring
        int fresh = 0;                             // slabs of this image that are known to be there
        uint32_t phase = 0;                        // parity of the ring's next slab to wait for
        int wait_slot = 0;
        auto next_of = [&](int x) { return x + 1 == p.b_stages ? 0 : x + 1; };
        for (int it = 0; it < n_kt && ok; ++it) {
          for (; fresh < 3 && ok; ++fresh) {
            ok = mbar_wait_suspend(full_b + 8 * wait_slot, phase);
            wait_slot = next_of(wait_slot);
            if (wait_slot == 0) phase ^= 1;
          }
          ok = ok && mbar_wait_suspend(full_a + 8 * sa, pa);
          if (!ok) break;
          tc_fence_after();
          const int slot1 = next_of(slot), slot2 = next_of(slot1);
          const uint64_t d[3] = {b_base + b_inc * static_cast<uint64_t>(slot), b_base + b_inc * static_cast<uint64_t>(slot1),
                                 b_base + b_inc * static_cast<uint64_t>(slot2)};
#pragma unroll
          for (int r = 0; r < 3; ++r) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              // kernel row r reads the gradient (1 - r) map rows further on
              constexpr int kSteps = kTileK / 16;
              const int step = kSteps + kk + (1 - r) * SLAB;       // K-steps from the start of slab kin
              umma_bf16(tmem_base + r * p.acc_n, da + static_cast<uint64_t>(kk * 2),
                        d[step / kSteps] + static_cast<uint64_t>((step % kSteps) * 128), idesc, kk > 0 ? 1u : accum);
            }
          }
          umma_commit(empty_a + 8 * sa);
          umma_commit(empty_b + 8 * slot);
          accum = 1;
          fresh = 2;
          slot = slot1;
          if (++kin == p.tiles_per_img || it + 1 == n_kt) {      // the image's last two slabs are done with as well
            umma_commit(empty_b + 8 * slot);
            slot = next_of(slot);
            umma_commit(empty_b + 8 * slot);
            slot = next_of(slot);
            kin = 0;
            fresh = 0;
          }
          if (++sa == p.a_stages) { sa = 0; pa ^= 1; da = a_base; } else { da += a_inc; }
        }
      } else
      for (int it = 0; it < n_kt; ++it) {
#ifdef SURGEON_DW_STATS
        const long long c0 = clock64();
        ok = mbar_wait_suspend(full_b + 8 * sb, pb);
        const long long c1 = clock64();
        ok = ok && (PAIR ? mbar_wait_suspend_cluster(full_a + 8 * sa, pa) : mbar_wait_suspend(full_a + 8 * sa, pa));
        st_g += c1 - c0; st_a += clock64() - c1;
#else
        ok = mbar_wait_suspend(full_b + 8 * sb, pb) &&
             (PAIR ? mbar_wait_suspend_cluster(full_a + 8 * sa, pa) : mbar_wait_suspend(full_a + 8 * sa, pa));
#endif
        if (!ok) break;
        tc_fence_after();
        if (TG) {
          if (n_acc_here == 1) umma_ktile_tg<1>(tmem_base, p.acc_n, da, db + first_row, acc_inc, idesc, accum);
          else if (n_acc_here == 2) umma_ktile_tg<2>(tmem_base, p.acc_n, da, db + first_row, acc_inc, idesc, accum);
          else umma_ktile_tg<3>(tmem_base, p.acc_n, da, db + first_row, acc_inc, idesc, accum);
        } else
        if (n_acc_here == 1) umma_ktile<1, kStep, PAIR>(tmem_base, p.acc_n, da, db, acc_inc, idesc, accum);
        else if (n_acc_here == 2) umma_ktile<2, kStep, PAIR>(tmem_base, p.acc_n, da, db, acc_inc, idesc, accum);
        else if (n_acc_here == 3) umma_ktile<3, kStep, PAIR>(tmem_base, p.acc_n, da, db, acc_inc, idesc, accum);
        else umma_ktile<4, kStep, PAIR>(tmem_base, p.acc_n, da, db, acc_inc, idesc, accum);
        if (PAIR) { umma_commit_pair(empty_a + 8 * sa); umma_commit_pair(empty_b + 8 * sb); }
        else { umma_commit(empty_a + 8 * sa); umma_commit(empty_b + 8 * sb); }
        accum = 1;
        if (++sa == p.a_stages) { sa = 0; pa ^= 1; da = a_base; } else { da += a_inc; }
        if (++sb == p.b_stages) { sb = 0; pb ^= 1; db = b_base; } else { db += b_inc; }
      }
      if (!ok) { fail = 1; atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT)); }
#ifdef SURGEON_DW_STATS
      atomicAdd(reinterpret_cast<unsigned long long*>(status) + 4, static_cast<unsigned long long>(st_g));
      atomicAdd(reinterpret_cast<unsigned long long*>(status) + 5, static_cast<unsigned long long>(st_a));
      atomicAdd(reinterpret_cast<unsigned long long*>(status) + 6, static_cast<unsigned long long>(clock64() - st_begin));
      atomicAdd(reinterpret_cast<unsigned long long*>(status) + 7, static_cast<unsigned long long>(n_kt));
#endif
      if (PAIR) umma_commit_pair(acc_bar);
      else umma_commit(acc_bar);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ================= gradient tiles by TMA =================
    if (lane == 0) {
      pdl_wait();                                      // the bf16 gradient copy is complete
      int sb = 0;
      uint32_t round = 0;
      int img = 0, kin = 0;                            // conv: image and K-tile within it
      if (MODE != 0) { img = kt_begin / p.tiles_per_img; kin = kt_begin - img * p.tiles_per_img; }
      if (TG) {
        // Per K-tile (slabs: one more before and behind the K-tiles of an image): the boxes of 64 channels
        // and so many map rows, from row y on, of the CTA's units.
        const int per_unit = (p.acc_n + 63) / 64;
        const int tg_col = n_tile / p.upt, tg_o = (n_tile - tg_col * p.upt) * p.acc_n;   // TG >= 2
        const uint32_t slab_bytes = static_cast<uint32_t>(p.k_rows) * 128u;
        bool ok = true;
        for (int it = 0; it < n_kt && ok;) {
          const int n_here = min(n_kt - it, p.tiles_per_img - kin);
          for (int q = kin; q < kin + n_here + (SLAB ? 2 : 0); ++q) {
            if (round > 0 && !mbar_wait_suspend(empty_b + 8 * sb, (round - 1) & 1)) {
              fail = 1;
              atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
              ok = false;
              break;
            }
            const uint32_t b_addr = smem_u32(b_ring + sb * b_stage_bytes);
            if (TG == 1) {
              mbar_arrive_expect_tx(full_b + 8 * sb, static_cast<uint32_t>(n_acc_here * per_unit) * p.box_bytes);
              for (int a = 0; a < n_acc_here; ++a) {
                const int u = u0 + a, tap = u / p.upt, r = tap / p.kw;
                for (int j = 0; j < per_unit; ++j)
                  tma_load_4d(b_addr + a * p.unit_bytes + j * slab_bytes, &grad_map, (u - tap * p.upt) * p.acc_n + 64 * j,
                              p.pad - (tap - r * p.kw), q * p.map_rows + p.pad - r, img, full_b + 8 * sb);
              }
            } else {
              mbar_arrive_expect_tx(full_b + 8 * sb, static_cast<uint32_t>(per_unit) * p.box_bytes);
              const int y = SLAB ? (q - 1) * p.map_rows : q * p.map_rows + p.pad - (p.kh - 1);
              for (int j = 0; j < per_unit; ++j)
                tma_load_4d(b_addr + j * slab_bytes, &grad_map, tg_o + 64 * j, p.pad - tg_col, y, img, full_b + 8 * sb);
            }
            if (++sb == p.b_stages) { sb = 0; ++round; }
          }
          it += n_here;
          kin = 0;
          ++img;
        }
      } else
      for (int it = 0; it < n_kt; ++it) {
        if (round > 0 && !mbar_wait_suspend(empty_b + 8 * sb, (round - 1) & 1)) {
          fail = 1;
          atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
          break;
        }
        const uint32_t b_addr = smem_u32(b_ring + sb * b_stage_bytes);
        // rank 0 announces the bytes of both CTAs' loads of this tile
        if (cta_rank == 0)
          mbar_arrive_expect_tx(full_b + 8 * sb, static_cast<uint32_t>(n_acc_here * p.acc_n) * 128u);
        if (MODE == 0) {
          if (PAIR) {
            for (int a = 0; a < p.n_acc; ++a)
              for (int g = 0; g < acc_rows / 64; ++g)
                tma_load_2d_pair(b_addr + a * acc_rows * 128 + g * (kTileK * 128), &grad_map,
                                 o0 + a * p.acc_n + static_cast<int>(cta_rank) * acc_rows + g * 64,
                                 (kt_begin + it) * kTileK, full_b + 8 * sb);
          } else {
            for (int g = 0; g < p.n_cols / 64; ++g)
              tma_load_2d(b_addr + g * (kTileK * 128), &grad_map, o0 + g * 64, (kt_begin + it) * kTileK,
                          full_b + 8 * sb);
          }
        } else {
          const int p0 = kin * kTileK;
          for (int a = 0; a < n_acc_here; ++a) {
            // unit -> tap and channel range; the copy holding the tap's column shift, and the
            // tap's row shift as an offset along the flattened map
            const int u = u0 + a;
            const int tap = u / p.upt;
            const int o_lo = (u - tap * p.upt) * p.acc_n;
            int copy = tap, x = p0;
            if (p.row_shift) {
              const int r = tap / p.kw;
              copy = tap - r * p.kw;
              x = p0 + (p.pad - r) * p.in_w;
            }
            const int grow = copy * p.o_real + o_lo + static_cast<int>(cta_rank) * acc_rows;
            if (PAIR) tma_load_3d_pair(b_addr + a * acc_rows * 128, &grad_map, x, grow, img, full_b + 8 * sb);
            else tma_load_3d(b_addr + a * acc_rows * 128, &grad_map, x, grow, img, full_b + 8 * sb);
          }
          if (++kin == p.tiles_per_img) { kin = 0; ++img; }
        }
        if (++sb == p.b_stages) { sb = 0; ++round; }
      }
    }
    __syncwarp();
  } else {
    // ================= producers =================
    // Group g (warps 2 + 8g .. 9 + 8g) rebuilds the K-tiles g, g + kGroups, ... of this CTA's range.  A lane
    // owns one run of 32 consecutive elements per tile (linear: 32 channels of one row t; conv: 32
    // positions of one channel) = 64 bytes of the operand tile.
    const int pw = warp - 2;
    const int wg = pw >> 3, w8 = pw & 7;
    int row, part;                       // tile row and which run of the row
    if (MODE == 0) { row = 8 * w8 + static_cast<int>(lane >> 2); part = lane & 3; }   // k-row, 32-ch quarter
    else { row = 16 * w8 + static_cast<int>(lane >> 1); part = lane & 1; }            // channel, 32-pos half
    const uint32_t xr = row & 7;
    const uint32_t y = (MODE == 0) ? (part & 1) * 4 : part * 4;     // first 16-byte chunk of the run
    const uint32_t rowbase = (MODE == 0) ? (part >> 1) * (kTileK * 128) + row * 128 : row * 128;
    // per-warp staging of the packed values of a tile's rows (after the two rings)
    unsigned char* stg = b_ring + p.b_stages * b_stage_bytes + pw * kStageBytesPerWarp;
    const uint32_t n_keep = static_cast<uint32_t>(__ldg(p.n_keep_ptr));   // packed values in the store
    const bool few = n_keep <= p.few_keep;
    // ring position of this group's tile `it` (= it % a_stages) and how often it has wrapped
    int sa = wg % p.a_stages;
    uint32_t round = wg / p.a_stages;
    auto wait_stage = [&]() -> bool {
      if (round > 0 && lane == 0 && !mbar_wait_suspend(empty_a + 8 * sa, (round - 1) & 1)) {
        fail = 1;                                  // one lane polls; the warp follows
        atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
      }
      __syncwarp();
      return fail == 0;
    };
    auto next_stage = [&]() {
      sa += kGroups;
      while (sa >= p.a_stages) { sa -= p.a_stages; ++round; }
    };
    if (MODE != 0 && 16 * w8 >= rows_here) {
      // The warp's 16 rows hold no channel (the channels are spread evenly over the row tiles,
      // so every tile of a layer has idle warps when C is not a multiple of 128): they stay zero
      // in every stage, and the warp only keeps the barrier counts whole.
      for (int st = 0; st < p.a_stages; ++st) {
        unsigned char* dst_row = smem + st * kATileBytes + rowbase;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<uint4*>(dst_row + (((y + q) ^ xr) << 4)) = make_uint4(0, 0, 0, 0);
      }
      for (int it = wg; it < n_kt; it += kGroups) {
        if (!wait_stage()) break;
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) { if (PAIR) mbar_arrive_rank0(full_a + 8 * sa); else mbar_arrive(full_a + 8 * sa); }
        next_stage();
      }
    } else if (MODE == 2) {
      // 1x1 stride-2 conv: the run's 32 output positions sample every other element of every
      // other input row.  Per output-row segment: 64 bitmap bits from the segment's first input
      // element, the even ones are the segment's bits; a kept element's place in the packed
      // vector counts the odd (skipped) bits before it as well.
      for (int it = wg; it < n_kt; it += kGroups) {
        const int kt = kt_begin + it;
        const int img = kt / p.tiles_per_img;
        const int q0 = (kt - img * p.tiles_per_img) * kTileK + 32 * part;     // first output position
        const int c = c0 + row;
        int left = (row < rows_here) ? min(32, p.T - q0) : 0;
        if (!wait_stage()) break;
        unsigned char* dst_row = smem + sa * kATileBytes + rowbase;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<uint4*>(dst_row + (((y + q) ^ xr) << 4)) = make_uint4(0, 0, 0, 0);
        const long long plane = (static_cast<long long>(img) * p.C + c) * p.in_hw;
        int oy = q0 / p.ow, ox = q0 - oy * p.ow;
        int b0 = 0;                                    // position of the segment inside the run
        while (left > 0) {
          const int seg = min(left, p.ow - ox);
          const long long j = plane + static_cast<long long>(2 * oy) * p.in_w + 2 * ox;
          const long long blk = j >> kBlockShift;
          const long long wi = j >> 5;
          uint32_t rank = __ldg(offsets + blk);
          for (long long w = blk * kBlockWords; w < wi; ++w) rank += __popc(__ldg(bitmap + w));
          const uint32_t w0 = __ldg(bitmap + wi);
          const uint32_t w1 = (wi + 1 < p.n_words) ? __ldg(bitmap + wi + 1) : 0u;
          const uint32_t w2 = (wi + 2 < p.n_words) ? __ldg(bitmap + wi + 2) : 0u;
          const uint32_t sh = static_cast<uint32_t>(j & 31);
          rank += __popc(w0 & ((1u << sh) - 1u));
          unsigned long long win = (static_cast<unsigned long long>(__funnelshift_r(w1, w2, sh)) << 32) |
                                   __funnelshift_r(w0, w1, sh);
          // even bits of the window -> the segment's bits
          unsigned long long e = win & 0x5555555555555555ull;
          e = (e | (e >> 1)) & 0x3333333333333333ull;
          e = (e | (e >> 2)) & 0x0F0F0F0F0F0F0F0Full;
          e = (e | (e >> 4)) & 0x00FF00FF00FF00FFull;
          e = (e | (e >> 8)) & 0x0000FFFF0000FFFFull;
          e = (e | (e >> 16)) & 0x00000000FFFFFFFFull;
          uint32_t ev = static_cast<uint32_t>(e);
          ev = seg >= 32 ? ev : (ev & ((1u << seg) - 1u));
          // packed places of the kept samples are not contiguous (skipped odd elements lie
          // between them): eight loads in flight per round
          while (ev) {
            uint32_t vv[8];
            uint32_t e2 = ev;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int i = e2 ? __ffs(e2) - 1 : 0;
              vv[u] = ld_packed<DT>(values, rank + __popcll(win & ((1ull << (2 * i)) - 1ull)), e2 != 0);
              e2 &= e2 - 1;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              if (ev) {
                const int b = b0 + __ffs(ev) - 1;
                ev &= ev - 1;
                const unsigned short h = (DT == 0) ? to_bf16_bits(__uint_as_float(vv[u]))
                                                   : static_cast<unsigned short>(vv[u]);
                *reinterpret_cast<unsigned short*>(dst_row + (((y + (b >> 3)) ^ xr) << 4) + ((b & 7) << 1)) = h;
              }
            }
          }
          b0 += seg; left -= seg; ox = 0; ++oy;
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) { if (PAIR) mbar_arrive_rank0(full_a + 8 * sa); else mbar_arrive(full_a + 8 * sa); }
        next_stage();
      }
    } else if (MODE == 3) {
      // 1x1 stride 2: a K-tile is 64 / slot_w output rows, each at a multiple of slot_w positions: the lane's run is a part
      // of one row (slot_w 32 and 64), two rows or four.  A row's positions are every other element of every other input
      // row: the places of its kept ones count the elements between them.
      const bool many = n_keep > p.many_keep;
      auto rebuild = [&](auto segments) {
        constexpr int SEGS = decltype(segments)::value, NE = 32 / SEGS;
        struct Raw {
          uint32_t base, j, n;                         // kept count before the block; first element; elements that exist
          uint4 q;                                     // the block's words
          uint2 after;                                 // and the two behind it
        };
        auto fetch = [&](int kt, Raw (&raw)[SEGS]) {
          const int img = kt / p.tiles_per_img, kin = kt - img * p.tiles_per_img;
          const int x0 = SEGS == 1 ? (32 * part) & (p.slot_w - 1) : 0;
          const int ix = 2 * x0, n_row = max(0, min(NE, (p.in_w - ix + 1) >> 1));
          const int y0 = kin * p.map_rows + 32 * part / p.slot_w;
#pragma unroll
          for (int i = 0; i < SEGS; ++i) {
            Raw& r = raw[i];
            const int iy = 2 * (y0 + i);
            r.n = row < rows_here && iy < p.in_h ? n_row : 0;
            r.base = 0; r.q = make_uint4(0, 0, 0, 0); r.after = make_uint2(0, 0);
            r.j = ((static_cast<uint32_t>(img) * p.C + (c0 + row)) * p.in_h + iy) * p.in_w + ix;
            if (r.n > 0) {
              const uint32_t blk = r.j >> kBlockShift, w0 = blk * kBlockWords, n_words = static_cast<uint32_t>(p.n_words);
              r.base = __ldg(offsets + blk);
              if (blk != p.partial_blk) {
                r.q = __ldg(reinterpret_cast<const uint4*>(bitmap) + blk);
                if ((r.j & 64u) && w0 + 4 < n_words) {
                  if (w0 + 5 < n_words) r.after = __ldg(reinterpret_cast<const uint2*>(bitmap + w0 + 4));
                  else r.after.x = __ldg(bitmap + w0 + 4);
                }
              } else {                                 // the last, partial block of the bitmap
                r.q.x = __ldg(bitmap + w0);
                r.q.y = (w0 + 1 < n_words) ? __ldg(bitmap + w0 + 1) : 0u;
                r.q.z = (w0 + 2 < n_words) ? __ldg(bitmap + w0 + 2) : 0u;
                r.q.w = (w0 + 3 < n_words) ? __ldg(bitmap + w0 + 3) : 0u;
              }
            }
          }
        };
        constexpr bool kAhead = SEGS <= 2;             // (four rows' words would take 36 registers)
        Raw cur[SEGS];
        if (kAhead && wg < n_kt) fetch(kt_begin + wg, cur);
        for (int it = wg; it < n_kt; it += kGroups) {
          Raw nxt[SEGS];
          if (!kAhead) fetch(kt_begin + it, cur);
          else if (it + kGroups < n_kt) fetch(kt_begin + it + kGroups, nxt);
          // place of the first element's value, and the bits of the row's elements and of those between them
          uint32_t rank[SEGS], win[SEGS][2];
#pragma unroll
          for (int i = 0; i < SEGS; ++i) {
            const Raw& r = cur[i];
            const uint32_t wq = (r.j >> 5) & 3u, sh = r.j & 31u;
            rank[i] = r.base + (wq > 0 ? __popc(r.q.x) : 0u) + (wq > 1 ? __popc(r.q.y) : 0u) + (wq > 2 ? __popc(r.q.z) : 0u);
            const uint32_t w0 = wq == 0 ? r.q.x : (wq == 1 ? r.q.y : (wq == 2 ? r.q.z : r.q.w));
            const uint32_t w1 = wq == 0 ? r.q.y : (wq == 1 ? r.q.z : (wq == 2 ? r.q.w : r.after.x));
            const uint32_t w2 = wq == 0 ? r.q.z : (wq == 1 ? r.q.w : (wq == 2 ? r.after.x : r.after.y));
            rank[i] += __popc(w0 & ((1u << sh) - 1u));
            win[i][0] = __funnelshift_r(w0, w1, sh);
            win[i][1] = SEGS == 1 ? __funnelshift_r(w1, w2, sh) : 0u;
            const uint32_t bits = 2 * r.n;
            if (bits < 32) { win[i][0] &= (1u << bits) - 1u; win[i][1] = 0; }
            else if (bits < 64) win[i][1] &= (1u << (bits - 32)) - 1u;
          }
          unsigned char* dst_row = smem + sa * kATileBytes + rowbase;
          if (many) {
            // A lane per element, run by run, so that a load's values lie side by side.  (A lane's own loads touch a
            // cache line each, more lines than the L1 beside 200 KB of tiles holds until their last use.)
            // The lanes of segment i ask for their numbers in the register that lane 32 / SEGS * i + ... holds: a run's
            // segments are spread over the lanes first.
            if (!wait_stage()) break;
            constexpr int RUNS = 32 / SEGS;                            // runs per round
            const int seg = static_cast<int>(lane) / NE, e2 = 2 * (static_cast<int>(lane) % NE);
#pragma unroll
            for (int round_no = 0; round_no < SEGS; ++round_no) {
              // lane RUNS * i + k: segment i of run RUNS * round_no + k
              uint32_t at = 0, wa = 0, wb = 0;
#pragma unroll
              for (int i = 0; i < SEGS; ++i) {
                const int from = RUNS * round_no + static_cast<int>(lane) % RUNS;
                const uint32_t x = SEGS == 1 ? rank[i] : __shfl_sync(0xFFFFFFFFu, rank[i], from);
                const uint32_t y0 = SEGS == 1 ? win[i][0] : __shfl_sync(0xFFFFFFFFu, win[i][0], from);
                if (static_cast<int>(lane) / RUNS == i) { at = x; wa = y0; }
              }
              if (SEGS == 1) wb = win[0][1];
#pragma unroll 1
              for (int l0 = 0; l0 < RUNS; l0 += 8) {
                uint32_t v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const int from = RUNS * seg + l0 + u;
                  const uint32_t w0 = __shfl_sync(0xFFFFFFFFu, wa, from);
                  uint32_t idx = __shfl_sync(0xFFFFFFFFu, at, from), on;
                  if (SEGS == 1) {
                    const unsigned long long w = w0 | (static_cast<unsigned long long>(__shfl_sync(0xFFFFFFFFu, wb, from)) << 32);
                    idx += __popcll(w & ((1ull << e2) - 1ull));
                    on = static_cast<uint32_t>(w >> e2) & 1u;
                  } else {
                    idx += __popc(w0 & ((1u << e2) - 1u));
                    on = (w0 >> e2) & 1u;
                  }
                  v[u] = ld_packed<DT>(values, idx, on);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                  const int run = RUNS * round_no + l0 + u, rr = 16 * w8 + (run >> 1);     // whose: its tile row, and which half of it
                  unsigned char* to = smem + sa * kATileBytes + rr * 128 +
                                      ((((run & 1) * 4 + (static_cast<int>(lane) >> 3)) ^ (rr & 7)) << 4) + (lane & 7) * 2;
                  *reinterpret_cast<unsigned short*>(to) =
                      DT == 0 ? to_bf16_bits(__uint_as_float(v[u])) : static_cast<unsigned short>(v[u]);
                }
              }
            }
          } else {
            uint32_t v[32];
#pragma unroll
            for (int i = 0; i < SEGS; ++i) {
              uint32_t idx = rank[i];
#pragma unroll
              for (int e = 0; e < NE; ++e) {
                const uint32_t w = win[i][e >> 4], bit = 1u << (2 * (e & 15));
                v[i * NE + e] = ld_packed<DT>(values, idx, w & bit);
                if (w & bit) ++idx;
                if (w & (bit << 1)) ++idx;
              }
            }
            uint4 chunk[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t o[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const uint32_t lo = v[8 * q + 2 * e], hi = v[8 * q + 2 * e + 1];
                o[e] = DT == 0 ? pack_bf16x2(__uint_as_float(lo), __uint_as_float(hi)) : lo | (hi << 16);
              }
              chunk[q] = make_uint4(o[0], o[1], o[2], o[3]);
            }
            if (!wait_stage()) break;
#pragma unroll
            for (int q = 0; q < 4; ++q)
              *reinterpret_cast<uint4*>(dst_row + (((y + q) ^ xr) << 4)) = chunk[q];
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(full_a + 8 * sa);
          next_stage();
          if (kAhead) {
#pragma unroll
            for (int i = 0; i < SEGS; ++i) cur[i] = nxt[i];
          }
        }
      };
      if (p.slot_w >= 32) rebuild(std::integral_constant<int, 1>{});
      else if (p.slot_w == 16) rebuild(std::integral_constant<int, 2>{});
      else rebuild(std::integral_constant<int, 4>{});
    } else {
      // Flat index of the lane's run in the group's first tile, advanced by two tiles per round
      // without multiplications: linear j = t * C + c; conv j = (img * C + c) * T + position.
      const int kt_first = kt_begin + wg;
      long long j_run;                     // linear: flat index; conv: flat index of the row's image plane
      long long t_row = 0;                 // linear: row t of the run
      int kin = 0;                         // conv: K-tile within the image
      int n_run;                           // linear: channels of the run that exist (constant)
      if (MODE == 0) {
        const int c = c0 + 32 * part;
        n_run = max(0, min(32, p.C - c));
        t_row = static_cast<long long>(kt_first) * kTileK + row;
        j_run = t_row * p.C + c;
      } else {
        const int img = kt_first / p.tiles_per_img;
        kin = kt_first - img * p.tiles_per_img;
        n_run = (row < rows_here) ? 1 : 0;
        j_run = (static_cast<long long>(img) * p.C + (c0 + row)) * p.T;
      }
      const long long j_step = (MODE == 0) ? static_cast<long long>(kGroups) * kTileK * p.C : static_cast<long long>(p.C) * p.T;
      auto fetch = [&]() {                 // metadata of the run at the current position
        WordRaw r;
        r.base = 0; r.next = 0; r.words = make_uint4(0, 0, 0, 0); r.j = 0; r.nvalid = 0;
        long long j;
        int nvalid;
        if (MODE == 0) {
          nvalid = (t_row < p.T) ? n_run : 0;
          j = j_run;
        } else {
          const int pp = kin * (TG ? p.kpos : kTileK) + 32 * part;
          nvalid = n_run ? max(0, min(TG ? min(32, p.kpos - 32 * part) : 32, p.T - pp)) : 0;
          j = j_run + pp;
        }
        if (nvalid > 0) {
          r.nvalid = static_cast<uint32_t>(nvalid);
          r.j = static_cast<uint32_t>(j);
          const long long blk = j >> kBlockShift;
          const long long wi = j >> 5;
          r.base = __ldg(offsets + blk);
          if (static_cast<unsigned long long>(blk) != p.partial_blk) {
            r.words = __ldg(reinterpret_cast<const uint4*>(bitmap) + blk);
          } else {                                   // the last, partial block of the bitmap
            const long long w0 = blk * kBlockWords;
            r.words.x = __ldg(bitmap + w0);
            r.words.y = (w0 + 1 < p.n_words) ? __ldg(bitmap + w0 + 1) : 0u;
            r.words.z = (w0 + 2 < p.n_words) ? __ldg(bitmap + w0 + 2) : 0u;
            r.words.w = (w0 + 3 < p.n_words) ? __ldg(bitmap + w0 + 3) : 0u;
          }
          if ((r.j & 31u) && wi + 1 < p.n_words) r.next = __ldg(bitmap + wi + 1);
        }
        return r;
      };
      auto advance = [&]() {               // two K-tiles on
        if (MODE == 0) { t_row += kGroups * kTileK; j_run += j_step; }
        else {
          kin += kGroups;
          while (kin >= p.tiles_per_img) { kin -= p.tiles_per_img; j_run += j_step; }
        }
      };
      WordRaw cur = {};
      if (wg < n_kt) cur = fetch();
      for (int it = wg; it < n_kt; it += kGroups) {
        WordRaw nxt = {};
        advance();
        if (it + kGroups < n_kt) nxt = fetch();             // in flight while this tile is rebuilt
        // bits of the run and rank of its first kept element
        const uint32_t wq = (cur.j >> 5) & 3, sh = cur.j & 31;
        uint32_t rank = cur.base;
        rank += wq > 0 ? __popc(cur.words.x) : 0u;
        rank += wq > 1 ? __popc(cur.words.y) : 0u;
        rank += wq > 2 ? __popc(cur.words.z) : 0u;
        const uint32_t w0 = wq == 0 ? cur.words.x : (wq == 1 ? cur.words.y : (wq == 2 ? cur.words.z : cur.words.w));
        const uint32_t w1 = wq == 3 ? cur.next : (wq == 0 ? cur.words.y : (wq == 1 ? cur.words.z : cur.words.w));
        rank += __popc(w0 & ((1u << sh) - 1u));
        uint32_t bits = __funnelshift_r(w0, w1, sh);
        bits = cur.nvalid >= 32 ? bits : (bits & ((1u << cur.nvalid) - 1u));
        // ---- the packed values of the warp's rows -> shared memory, as bf16 ----
        // The lanes of a row (2 for conv, 4 for linear) hold consecutive runs, so a row's kept
        // values are one contiguous piece of the packed vector.  The warp copies every piece
        // with aligned 16-byte loads, lane by lane (coalesced; the lane-per-run loads they
        // replace touch a cache line per lane and saturate the L1 at low pruning ratios),
        // converting fp32 to bf16 on the way; each row has its own slot.
        constexpr int LPR = (MODE == 0) ? 4 : 2;              // lanes per row
        constexpr int RPW = 32 / LPR;                         // rows per warp
        constexpr int V = (DT == 0) ? 4 : 8;                  // packed values per 16-byte vector
        constexpr int VMAX = (32 * LPR + V - 1) / V + 1;      // vectors a row's piece can span
        constexpr int ITER = (RPW * VMAX + 31) / 32;
        constexpr int kSlot = 32 * LPR + 16;                  // bf16 values per row slot (piece + alignment slack)
        const uint32_t cnt = __popc(bits);
        uint4 chunk[4];
        // Dense tiles of fp32 activations (more than 55 % of the warp's 1024 elements kept) go
        // through the staging copy; for sparser ones the copy's fixed cost outweighs the
        // scattered loads it saves, and bf16 values (half as many cache lines per load) never
        // gain from it, so bf16 launches reserve no staging area.
        // Every run of the warp fully kept and its values 16-byte aligned: the layer that Eq. 7 gives
        // ratio 0 (there is one in every batch: the layer with the largest importance), or an
        // unpruned tensor.  The run is then 64 (128) consecutive bytes of the packed vector.
        const bool whole = __all_sync(0xFFFFFFFFu, bits == 0xFFFFFFFFu && (rank & static_cast<uint32_t>(V - 1)) == 0u);
        // Few elements per run (an eighth at most in the whole store; the fullest run of the warp decides): a loop
        // over the kept elements, whose values lie one behind the other (immediate offsets), scattered into a
        // zeroed run; some 12 instructions per element of the fullest run against 6 per position.  At 7 % kept
        // 91 -> 85 us (768 -> 2304 channels), at 10 % 107 -> 103 (256 -> 256); at a third 142 -> 158, hence the rule.
        const uint32_t most = few ? __reduce_max_sync(0xFFFFFFFFu, cnt) : 32u;
        if (most <= kFewMost) {
          constexpr int kFirst = 8;                           // loads in flight before the tile's place is free
          const unsigned char* src = reinterpret_cast<const unsigned char*>(values) + static_cast<size_t>(rank) * (DT == 0 ? 4 : 2);
          uint32_t first[kFirst];
#pragma unroll
          for (uint32_t u = 0; u < kFirst; ++u) first[u] = ld_packed<DT>(src, u, u < cnt);
          if (!wait_stage()) break;
          const uint32_t dst = smem_u32(smem + sa * kATileBytes + rowbase);
#pragma unroll
          for (int q = 0; q < 4; ++q)
            asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(dst + (((y + q) ^ xr) << 4)), "r"(0) : "memory");
          uint32_t m = bits;
          auto put = [&](uint32_t value, bool on) {
            const uint32_t e = __ffs(m) - 1;
            m &= m - 1;
            const unsigned short h = (DT == 0) ? to_bf16_bits(__uint_as_float(value)) : static_cast<unsigned short>(value);
            asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q st.shared.u16 [%0], %1;\n\t}"
                         ::"r"(dst + (((y + (e >> 3)) ^ xr) << 4) + ((e & 7) << 1)), "h"(h), "r"(static_cast<uint32_t>(on)) : "memory");
          };
#pragma unroll
          for (uint32_t u = 0; u < kFirst; ++u) put(first[u], u < cnt);
#pragma unroll 1
          for (uint32_t k = kFirst; k < most; k += 4) {
            uint32_t more[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) more[u] = ld_packed<DT>(src, k + u, k + u < cnt);
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) put(more[u], k + u < cnt);
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) { if (PAIR) mbar_arrive_rank0(full_a + 8 * sa); else mbar_arrive(full_a + 8 * sa); }
          next_stage();
          cur = nxt;
          continue;
        }
        const bool dense = !whole && DT == 0 && __reduce_add_sync(0xFFFFFFFFu, cnt) > 560u;
        if (whole) {
          if (DT == 0) {
            const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(values) + rank);
            float4 f[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) f[q] = __ldg(src + q);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              chunk[q].x = pack_bf16x2(f[2 * q].x, f[2 * q].y); chunk[q].y = pack_bf16x2(f[2 * q].z, f[2 * q].w);
              chunk[q].z = pack_bf16x2(f[2 * q + 1].x, f[2 * q + 1].y); chunk[q].w = pack_bf16x2(f[2 * q + 1].z, f[2 * q + 1].w);
            }
          } else {
            const uint4* src = reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned short*>(values) + rank);
#pragma unroll
            for (int q = 0; q < 4; ++q) chunk[q] = __ldg(src + q);
          }
        } else if (dense) {
        uint32_t seg_len = cnt + __shfl_xor_sync(0xFFFFFFFFu, cnt, 1);
        if (MODE == 0) seg_len += __shfl_xor_sync(0xFFFFFFFFu, seg_len, 2);
        const uint32_t seg_start = __shfl_sync(0xFFFFFFFFu, rank, lane & ~(LPR - 1));
        const uint32_t a0 = seg_start & ~static_cast<uint32_t>(V - 1);
        const uint32_t nvec = seg_len ? (seg_start + seg_len - a0 + V - 1) / V : 0u;
        __syncwarp();                                         // the previous tile's slot reads are done
#pragma unroll
        for (int i = 0; i < ITER; ++i) {
          const int t = static_cast<int>(lane) + 32 * i;
          const int r = min(t / VMAX, RPW - 1), v = t - (t / VMAX) * VMAX;
          const uint32_t a0_r = __shfl_sync(0xFFFFFFFFu, a0, r * LPR);
          const uint32_t nvec_r = __shfl_sync(0xFFFFFFFFu, nvec, r * LPR);
          if (t < RPW * VMAX && static_cast<uint32_t>(v) < nvec_r) {
            const uint32_t first = a0_r + static_cast<uint32_t>(v) * V;
            unsigned char* dst = stg + r * (kSlot * 2) + v * 16 / (DT == 0 ? 2 : 1);
            if (DT == 0) {
              const float* src = reinterpret_cast<const float*>(values) + first;
              float4 f;
              if (first + V <= n_keep) f = __ldg(reinterpret_cast<const float4*>(src));
              else {                                          // the vector that ends past the last value
                f.x = first < n_keep ? __ldg(src) : 0.0f;
                f.y = first + 1 < n_keep ? __ldg(src + 1) : 0.0f;
                f.z = first + 2 < n_keep ? __ldg(src + 2) : 0.0f;
                f.w = 0.0f;
              }
              *reinterpret_cast<uint2*>(dst) = make_uint2(pack_bf16x2(f.x, f.y), pack_bf16x2(f.z, f.w));
            } else {
              const unsigned short* src = reinterpret_cast<const unsigned short*>(values) + first;
              uint4 u;
              if (first + V <= n_keep) u = __ldg(reinterpret_cast<const uint4*>(src));
              else {
                uint32_t h[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) h[e] = first + e < n_keep ? static_cast<uint32_t>(__ldg(src + e)) : 0u;
                u = make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
              }
              *reinterpret_cast<uint4*>(dst) = u;
            }
          }
        }
        __syncwarp();
        // ---- the run as four 16-byte chunks of 8 elements, read from the row's slot ----
        const unsigned short* slot = reinterpret_cast<const unsigned short*>(
            stg + (lane / LPR) * (kSlot * 2)) + (rank - a0);
        uint32_t k = 0;                                       // kept elements of the run so far
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t v[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const uint32_t on = (bits >> (8 * q + e)) & 1u;
            v[e] = on ? static_cast<uint32_t>(slot[k]) : 0u;
            k += on;
          }
          chunk[q].x = v[0] | (v[1] << 16); chunk[q].y = v[2] | (v[3] << 16);
          chunk[q].z = v[4] | (v[5] << 16); chunk[q].w = v[6] | (v[7] << 16);
        }
        } else {
          // sparse: one predicated global load per element, all of a lane's loads independent
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t byte = (bits >> (8 * q)) & 0xFFu;
            uint32_t idx = rank + (q == 0 ? 0u : __popc(bits & ((1u << (8 * q)) - 1u)));
            uint32_t v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const uint32_t on = (byte >> e) & 1u;
              v[e] = ld_packed<DT>(values, idx, on != 0);
              idx += on;
            }
            if (DT == 0) {
              chunk[q].x = pack_bf16x2(__uint_as_float(v[0]), __uint_as_float(v[1]));
              chunk[q].y = pack_bf16x2(__uint_as_float(v[2]), __uint_as_float(v[3]));
              chunk[q].z = pack_bf16x2(__uint_as_float(v[4]), __uint_as_float(v[5]));
              chunk[q].w = pack_bf16x2(__uint_as_float(v[6]), __uint_as_float(v[7]));
            } else {
              chunk[q].x = v[0] | (v[1] << 16); chunk[q].y = v[2] | (v[3] << 16);
              chunk[q].z = v[4] | (v[5] << 16); chunk[q].w = v[6] | (v[7] << 16);
            }
          }
        }
        if (!wait_stage()) break;
        unsigned char* dst_row = smem + sa * kATileBytes + rowbase;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<uint4*>(dst_row + (((y + q) ^ xr) << 4)) = chunk[q];
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) { if (PAIR) mbar_arrive_rank0(full_a + 8 * sa); else mbar_arrive(full_a + 8 * sa); }
        next_stage();
        cur = nxt;
      }
    }
  }

  // ================= epilogue: TMEM -> scratch partial tile =================
  if (warp >= 2) {
    // a warp may read the 32 TMEM lanes of its quarter (warp % 4); the warps of a quarter take
    // the groups of 16 columns in turn
    // (MODE != 0) the tap of the accumulator at hand and its first channel; a column's place in the accumulator
    int tap = 0, o_acc = 0, rel = 16 * ((warp - 2) >> 2);
    if (MODE != 0) {
      const int u = TG >= 2 ? n_tile : u0;         // TG >= 2: accumulator a is kernel row a of this CTA's kernel column
      tap = u / p.upt;
      o_acc = (u - tap * p.upt) * p.acc_n;
    }
    const bool done = mbar_wait(acc_bar, 0, 64);
    tc_fence_after();
    if (done && !fail) {
      const int lane_grp = warp & 3;
      const long long first = static_cast<long long>(split) * p.O * p.C + c0 + lane_grp * 32;
      float* buf = reinterpret_cast<float*>(smem) + (warp - 2) * 512;      // (the rings are done with)
      const bool vec = (p.C & 3) == 0;             // (a row tile begins at a multiple of 16, and so a tile's end is one of 4)
      const int cols_here = n_acc_here * p.acc_n;
      for (int col = rel; col < cols_here; col += 16 * (kProdWarps / 4), rel += 16 * (kProdWarps / 4)) {
        uint32_t r[16];
        tmem_ld16(tmem_base + (static_cast<uint32_t>(lane_grp * 32) << 16) + col, r);
        int row0, n_ok;                   // first partial row of the 16 columns, how many exist
        if (MODE == 0) {
          row0 = o0 + col; n_ok = p.O - row0;
        } else {
          for (; rel >= p.acc_n; rel -= p.acc_n) {
            if (TG >= 2) tap += p.kw;
            else if ((o_acc += p.acc_n) == p.upt * p.acc_n) { o_acc = 0; ++tap; }
          }
          row0 = tap * p.o_real + o_acc + rel; n_ok = p.o_real - (o_acc + rel);
        }
        const long long at = first + static_cast<long long>(row0) * p.C;
        store_cols16(buf, r, partial + at, p.C, n_ok, rows_here - lane_grp * 32, vec, at,
                     static_cast<long long>(p.splits) * p.O * p.C, status);
      }
    } else if (!done && lane == 0) {
      atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync_all();          // neither CTA leaves while the pair's MMAs or arrivals may touch it
  if (warp == 0) {
    if (PAIR) tmem_dealloc_pair(tmem_base, p.tmem_cols);
    else tmem_dealloc(tmem_base, p.tmem_cols);
  }
}

// TG: out[img][position][channel] = g[img][channel][position], 64 channels x 64 positions per block through
// shared memory.  A thread reads four positions of two channels, so that it stores channel pairs.
__global__ void __launch_bounds__(256)
grad_transpose_bf16_kernel(const float* __restrict__ g, unsigned short* __restrict__ out,
                           long long blocks, DirectParams p, uint32_t* __restrict__ status) {
  prepass_begin(status);
  __shared__ uint32_t tile[64][33];                    // [position][channel pair]
  const int hw = p.oh * p.ow;
  const int pos_blocks = (hw + 63) >> 6, ch_blocks = (p.o_real + 63) >> 6;
  const int q = threadIdx.x & 15, pair = threadIdx.x >> 4;
  for (long long b = blockIdx.x; b < blocks; b += gridDim.x) {
    const int cb = static_cast<int>(b % ch_blocks);
    const long long t = b / ch_blocks;
    const int pb = static_cast<int>(t % pos_blocks);
    const long long img = t / pos_blocks;
    const int pos = pb * 64 + 4 * q;
    float4 v[2][2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int o = cb * 64 + 2 * (pair + 16 * i) + h;
        const float* src = g + (img * p.o_real + o) * hw + pos;
        float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (o < p.o_real) {
          if ((hw & 3) == 0 && pos < hw) x = __ldg(reinterpret_cast<const float4*>(src));
          else {
            x.x = pos < hw ? __ldg(src) : 0.0f;
            x.y = pos + 1 < hw ? __ldg(src + 1) : 0.0f;
            x.z = pos + 2 < hw ? __ldg(src + 2) : 0.0f;
            x.w = pos + 3 < hw ? __ldg(src + 3) : 0.0f;
          }
        }
        v[i][h] = x;
      }
    }
    __syncthreads();                                   // the previous block's rows are out
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int c2 = pair + 16 * i;
      tile[4 * q][c2] = pack_bf16x2(v[i][0].x, v[i][1].x);
      tile[4 * q + 1][c2] = pack_bf16x2(v[i][0].y, v[i][1].y);
      tile[4 * q + 2][c2] = pack_bf16x2(v[i][0].z, v[i][1].z);
      tile[4 * q + 3][c2] = pack_bf16x2(v[i][0].w, v[i][1].w);
    }
    __syncthreads();
    // 16 bytes (8 channels) per thread: 8 threads per position
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int row = (threadIdx.x >> 3) + 32 * i, c8 = threadIdx.x & 7;
      const int at = pb * 64 + row, o = cb * 64 + 8 * c8;
      if (at < hw && o < p.o_real)
        *reinterpret_cast<uint4*>(out + (img * hw + at) * p.o_real + o) =
            make_uint4(tile[row][4 * c8], tile[row][4 * c8 + 1], tile[row][4 * c8 + 2], tile[row][4 * c8 + 3]);
    }
  }
}

// Shifted bf16 copies of the output gradient of a k x k stride-1 convolution (Eq. 2 summed over
// input positions): out[img][tap * O + o][y' * W + x'] = g[img][o][y' + pad - r][x' + pad - s],
// zero where that lies outside the output map; tap = r * kw + s.  One thread writes 8 positions.
__global__ void __launch_bounds__(256)
grad_taps_bf16_kernel(const float* __restrict__ g, unsigned short* __restrict__ out,
                      long long chunks, DirectParams p, uint32_t* __restrict__ status) {
  prepass_begin(status);
  const int per_row = p.pitch >> 3;
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < chunks;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long rowi = i / per_row;              // img * taps * O + tap * O + o
    const int chunk = static_cast<int>(i - rowi * per_row);
    const int v = static_cast<int>(rowi % p.O);
    const long long img = rowi / p.O;
    const int tap = v / p.o_real, o = v - tap * p.o_real;
    const int r = tap / p.kw, sft = tap - r * p.kw;
    const float* src = g + (img * p.o_real + o) * static_cast<long long>(p.oh) * p.ow;
    int pos = chunk * 8;
    int yy = pos / p.in_w, xx = pos - yy * p.in_w;   // input position
    float f[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int y = yy + p.pad - r, x = xx + p.pad - sft;
      f[e] = (pos < p.T && y >= 0 && y < p.oh && x >= 0 && x < p.ow) ? __ldg(src + y * p.ow + x) : 0.0f;
      ++pos; ++xx;
      if (xx == p.in_w) { xx = 0; ++yy; }
    }
    uint4 w;
    w.x = pack_bf16x2(f[0], f[1]); w.y = pack_bf16x2(f[2], f[3]);
    w.z = pack_bf16x2(f[4], f[5]); w.w = pack_bf16x2(f[6], f[7]);
    *reinterpret_cast<uint4*>(out + rowi * p.pitch + chunk * 8) = w;
  }
}

// The same for rows a multiple of 8 wide, where only the KW column shifts are materialised:
// out[img][s * O + o][y * W + x'] = g[img][o][y][x' + pad - s] for the OH gradient rows y (zero
// where the column lies outside the output map).  One thread reads a window of 8 + KW - 1
// gradient values and writes 8 positions of every shift.
// The same copies for a same-padded convolution (odd KW, padding (KW - 1) / 2, output map = input
// map): the source of input position pos under tap (r, s) is the flat index
// pos + (pad - r) * W + (pad - s) of the output gradient's plane, so one thread reads a window of
// 8 + KW - 1 consecutive values for a row shift r and writes the KW column shifts from it; a value
// is dropped where the shifted column leaves the row.
template <int KW>
__global__ void __launch_bounds__(256)
grad_taps_same_bf16_kernel(const float* __restrict__ g, unsigned short* __restrict__ out,
                           long long items, DirectParams p, uint32_t* __restrict__ status) {
  prepass_begin(status);
  constexpr int H = (KW - 1) / 2;
  const int per_row = p.pitch >> 3;
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < items;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    long long t = i / per_row;
    const int chunk = static_cast<int>(i - t * per_row);
    const int r = static_cast<int>(t % p.kh);
    t /= p.kh;
    const int o = static_cast<int>(t % p.o_real);
    const long long img = t / p.o_real;
    const float* src = g + (img * p.o_real + o) * static_cast<long long>(p.T);
    const int pos0 = chunk * 8;
    const int yy0 = pos0 / p.in_w;
    int xx = pos0 - yy0 * p.in_w;
    const int base = pos0 + (p.pad - r) * p.in_w - H;      // flat index of w[0]
    float w[8 + 2 * H];
#pragma unroll
    for (int j = 0; j < 8 + 2 * H; ++j) {
      const int q = base + j;
      w[j] = (q >= 0 && q < p.T) ? __ldg(src + q) : 0.0f;
    }
    int xe[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      xe[e] = (pos0 + e < p.T) ? xx : -64;                 // past the map: no column is valid
      if (++xx == p.in_w) xx = 0;
    }
#pragma unroll
    for (int sft = 0; sft < KW; ++sft) {
      float f[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int x = xe[e] + H - sft;
        f[e] = (x >= 0 && x < p.in_w) ? w[e + 2 * H - sft] : 0.0f;
      }
      uint4 v;
      v.x = pack_bf16x2(f[0], f[1]); v.y = pack_bf16x2(f[2], f[3]);
      v.z = pack_bf16x2(f[4], f[5]); v.w = pack_bf16x2(f[6], f[7]);
      const long long rowi = (img * p.taps + r * KW + sft) * p.o_real + o;
      *reinterpret_cast<uint4*>(out + rowi * p.pitch + chunk * 8) = v;
    }
  }
}

// SAME: padding (KW - 1) / 2 with KW odd, so the output map is as wide as the input (a multiple of
// 8): the 8 elements of a chunk are two aligned 16-byte loads, only the halo is fetched singly.
template <int KW, bool SAME>
__global__ void __launch_bounds__(256)
grad_cols_bf16_kernel(const float* __restrict__ g, unsigned short* __restrict__ out,
                      long long chunks, DirectParams p, uint32_t* __restrict__ status) {
  prepass_begin(status);
  const int per_row = p.in_w >> 3;                     // chunks per map row
  const int per_plane = p.pitch >> 3;                  // pitch = OH * W
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < chunks;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    const long long plane = i / per_plane;             // img * O + o
    const int chunk = static_cast<int>(i - plane * per_plane);
    const int y = chunk / per_row;
    const int x0 = (chunk - y * per_row) * 8;
    const long long img = plane / p.o_real;
    const int o = static_cast<int>(plane - img * p.o_real);
    const float* src = g + (plane * p.oh + y) * static_cast<long long>(p.ow);
    float f[8 + KW - 1];                               // f[j] = g[y][x0 + pad - (KW - 1) + j]
    if (SAME) {
      constexpr int H = (KW - 1) / 2;                  // f[j] = g[y][x0 - H + j]
      const float4 a = __ldg(reinterpret_cast<const float4*>(src + x0));
      const float4 b = __ldg(reinterpret_cast<const float4*>(src + x0 + 4));
      f[H] = a.x; f[H + 1] = a.y; f[H + 2] = a.z; f[H + 3] = a.w;
      f[H + 4] = b.x; f[H + 5] = b.y; f[H + 6] = b.z; f[H + 7] = b.w;
#pragma unroll
      for (int j = 0; j < H; ++j) {
        const int xl = x0 - H + j, xr = x0 + 8 + j;
        f[j] = xl >= 0 ? __ldg(src + xl) : 0.0f;
        f[H + 8 + j] = xr < p.ow ? __ldg(src + xr) : 0.0f;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8 + KW - 1; ++j) {
        const int x = x0 + p.pad - (KW - 1) + j;
        f[j] = (x >= 0 && x < p.ow) ? __ldg(src + x) : 0.0f;
      }
    }
#pragma unroll
    for (int sft = 0; sft < KW; ++sft) {
      const int b = KW - 1 - sft;                      // element e of shift sft is f[e + b]
      uint4 w;
      w.x = pack_bf16x2(f[b], f[b + 1]); w.y = pack_bf16x2(f[b + 2], f[b + 3]);
      w.z = pack_bf16x2(f[b + 4], f[b + 5]); w.w = pack_bf16x2(f[b + 6], f[b + 7]);
      unsigned short* dst = out + ((img * KW + sft) * p.o_real + o) * static_cast<long long>(p.pitch) +
                            static_cast<long long>(chunk) * 8;
      *reinterpret_cast<uint4*>(dst) = w;
    }
  }
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                              CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                              CUtensorMapFloatOOBfill);

}  // namespace

// Shared memory: the staging area of the packed values (fp32 activations only), the gradient
// ring (as many tiles as fit beside four activation tiles, up to 4; slabs up to 8, beside three activation tiles and up
// to 6 for fp32 activations), then as many activation tiles as fit (up to 8).
static bool size_rings(DirectParams* p, int stage_bytes) {
  const int budget = 224 * 1024 - 1024 - stage_bytes;
  const int b_bytes = p->tg ? p->b_bytes : p->n_cols * (p->pair ? 64 : 128);
  // Slabs: a K-tile holds three, so two more are wanted under way.  Beside the staging area of fp32 activations a fourth
  // activation tile leaves room for one (the MMA thread waited 420-690 of 1700-2000 clocks a K-tile for them; 160 channels
  // on 32x32, 7 % kept, 173 -> 160 us, 320 on 16x16 148 -> 140); more than three under way take activation tiles for
  // nothing.  bf16 activations have no staging area, and the fourth tile is worth more to them (256 channels on 64x64,
  // batch 16, 70 % kept: 171 us, with three 174; 30 % kept 139 and 142).
  const bool slabs = p->tg >= 3, few_tiles = slabs && stage_bytes > 0;
  const int least = slabs ? 4 : 2, most = few_tiles ? 6 : (slabs ? kMaxBStages : 4);
  int b_stages = (budget - (few_tiles ? 3 : 4) * kATileBytes) / b_bytes;
  if (b_stages > most) b_stages = most;
  if (b_stages < least) b_stages = least;
  if (b_stages * b_bytes + 2 * kATileBytes > budget) return false;
  int a_stages = (budget - b_stages * b_bytes) / kATileBytes;
  if (a_stages > kMaxAStages) a_stages = kMaxAStages;
  if (a_stages < 2) return false;
  p->a_stages = a_stages; p->b_stages = b_stages;
  p->smem_bytes = a_stages * kATileBytes + b_stages * b_bytes + stage_bytes + 1024;
  return true;
}

static bool compute_plan_direct(const surgeon_layer_desc& d, bool transposed_ok, bool share, DirectParams* out) {
  DirectParams p{};
  if (d.kind == 0) {
    p.mode = 0;
    p.T = d.batch; p.imgs = 1;
    if (d.c_in % 8 != 0 || d.c_out % 8 != 0) return false;   // 16-byte units / TMA row pitch
  } else if (d.kind == 1 && d.kh == 1 && d.kw == 1 && d.stride == 1 && d.pad == 0) {
    p.mode = 1;
    p.T = d.h * d.w; p.imgs = d.batch;
  } else if (d.kind == 1 && d.kh == 1 && d.kw == 1 && d.stride == 2 && d.pad == 0 && transposed_ok && d.w <= 128 &&
             d.c_out % 8 == 0 && d.c_out >= 48) {
    p.mode = 3;                                    // rows of output positions at multiples of slot_w, the gradient transposed
    p.tg = 1;
    p.taps = p.kh = p.kw = 1;
    p.in_h = d.h; p.in_w = d.w;
    p.oh = (d.h + 1) / 2; p.ow = (d.w + 1) / 2;
    p.slot_w = 8;
    while (p.slot_w < p.ow) p.slot_w *= 2;
    p.map_rows = kTileK / p.slot_w;
    p.T = p.oh * p.slot_w; p.imgs = d.batch;
  } else if (d.kind == 1 && d.kh == 1 && d.kw == 1 && d.stride == 2 && d.pad == 0) {
    p.mode = 2;                                    // output positions; the input is sampled
    p.ow = (d.w - 1) / 2 + 1;
    p.T = ((d.h - 1) / 2 + 1) * p.ow; p.imgs = d.batch;
    p.in_w = d.w; p.in_hw = d.h * d.w;
  } else if (d.kind == 1 && d.stride == 1 && d.kh * d.kw > 1 && d.kh <= 7 && d.kw <= 7 &&
             d.pad < d.kh && d.pad < d.kw) {
    // k x k, stride 1: the sum runs over INPUT positions, and tap (r, s) multiplies the
    // activation with the output gradient shifted by (pad - r, pad - s).  The shifted copies
    // (zero outside the map) are stacked as kh*kw*O gradient channels, which makes this the 1x1
    // problem with that many output channels; the activation operand is never expanded.
    // 8-16 channels fill an eighth of the tile's rows here; as im2col rows (channels x taps) they
    // fill a whole tile, and the gradient is read once instead of through shifted copies
    // (16 -> 160 channels, 3x3 on 32x32, batch 200: 145 against 181 us).  Fewer channels still
    // are quicker here (3 channels: 94 against 110 us).
    if (d.c_in >= 8 && d.c_in <= 16) return false;
    p.mode = 1;
    p.taps = d.kh * d.kw;
    p.kh = d.kh; p.kw = d.kw; p.pad = d.pad; p.in_h = d.h; p.in_w = d.w;
    p.oh = d.h + 2 * d.pad - d.kh + 1; p.ow = d.w + 2 * d.pad - d.kw + 1;
    if (p.oh < 1 || p.ow < 1) return false;
    p.T = d.h * d.w; p.imgs = d.batch;
    // Rows a multiple of 8 wide: only the kw column shifts need copies; a row shift is a
    // 16-byte-aligned offset of the TMA coordinate along the flattened map (zero fill outside).
    p.row_shift = (d.w % 8 == 0 && (d.kw == 2 || d.kw == 3 || d.kw == 5 || d.kw == 7)) ? 1 : 0;
    // One transposed copy (see the top of the file): TMA needs rows of 16 bytes, and units of few channels would
    // leave most of a 64-channel box empty.
    if (transposed_ok && d.w <= 64 && d.c_out % 8 == 0 && d.c_out >= 48) {
      p.map_rows = kTileK / d.w < d.h ? kTileK / d.w : d.h;
      if (d.kh == 3 && d.kw == 3 && d.pad == 1 && (d.w == 16 || d.w == 32 || d.w == 64) && d.h * d.w >= kTileK)
        p.tg = d.w == 16 ? 3 : (d.w == 32 ? 4 : 5);
      else
        p.tg = d.w % 8 == 0 && d.kh <= 3 ? 2 : 1;
    }
  } else {
    return false;
  }
  if (p.taps == 0) p.taps = 1;
  p.o_real = d.c_out;
  if (static_cast<long long>(p.taps) * d.c_out > 2147483647LL / 256) return false;
  if (p.taps > 1 && d.c_out > 65535) return false;    // grid of the tap reduction
  p.C = d.c_in; p.O = p.taps * d.c_out;
  p.copies = p.tg ? 1 : (p.row_shift ? p.kw : p.taps);
  p.g_len = p.row_shift ? p.oh * p.in_w : p.T;         // elements per row of the bf16 gradient copy
  p.pitch = (p.mode == 0) ? p.O : (p.g_len + 7) / 8 * 8;
  p.m_tiles = (p.C + kTileM - 1) / kTileM;
  // conv: the channels are spread evenly over the row tiles, in units of a warp's 16 rows
  p.rows_per_tile = (p.mode == 0) ? kTileM : ((p.C + p.m_tiles - 1) / p.m_tiles + 15) / 16 * 16;
  // Two or more row tiles: CTA pairs (each CTA 128 rows, the pair shares every gradient tile).
  p.pair = (p.m_tiles >= 2 && use_pairs() && !p.tg) ? 1 : 0;
  if (p.pair) p.m_tiles = (p.m_tiles + 1) / 2 * 2;
  if (p.mode == 0 && p.pair) {
    // accumulators of 128 columns (each CTA of the pair loads a 64-column slab of each), up to four
    const int units = (p.O + 127) / 128;
    p.acc_n = 128;
    int best_pad = -1;
    for (int na = 4; na >= 1; --na) {
      const int padded = (units + na - 1) / na * na;
      if (best_pad < 0 || padded < best_pad) { best_pad = padded; p.n_acc = na; }
    }
  } else if (p.mode == 0) {
    // columns come in slabs of 64; per CTA two accumulators of 192 or 128 columns, or one small one
    const int g = (p.O + 63) / 64;
    if (g <= 4) { p.n_acc = 1; p.acc_n = g * 64; }
    else {
      const int t6 = (g + 5) / 6 * 6, t4 = (g + 3) / 4 * 4;
      p.n_acc = 2;
      p.acc_n = (t6 <= t4) ? 192 : 128;
    }
  } else {
    // Columns come in units: one tap's output channels are cut into `upt` accumulators of acc_n
    // columns (a multiple of 16 with the fewest padded columns, then the widest); a CTA holds up
    // to three units (<= 512 TMEM columns).
    int best_waste = -1;
    // (TG >= 2: the kh accumulators of a kernel column share the 512 columns; an MMA has at most 256)
    for (int c = p.tg >= 2 ? std::min(256, 512 / p.kh / 16 * 16) : 256; c >= 16; c -= 16) {
      const int upt = (p.o_real + c - 1) / c;
      const int waste = upt * c - p.o_real;
      if (best_waste < 0 || waste < best_waste) { best_waste = waste; p.acc_n = c; p.upt = upt; }
    }
    p.n_units = p.taps * p.upt;
    const int col_cap = 512;
    p.n_acc = 1;
    while (p.n_acc < 3 && p.n_acc < p.n_units && (p.n_acc + 1) * p.acc_n <= col_cap) ++p.n_acc;
    if (p.tg) {
      if (p.tg >= 2) p.n_acc = p.kh;
      p.kpos = p.map_rows * (p.mode == 3 ? p.slot_w : p.in_w);
      const int box_rows = p.tg == 2 ? p.map_rows + p.kh - 1 : p.map_rows;
      p.k_rows = p.tg == 2 ? box_rows * p.in_w + (kTileK - p.kpos) : kTileK;
      p.box_bytes = static_cast<unsigned>(box_rows * (p.mode == 3 ? p.slot_w : p.in_w)) * 128u;
      p.unit_bytes = (p.acc_n + 63) / 64 * p.k_rows * 128;
      p.b_bytes = p.tg == 1 ? p.n_acc * p.unit_bytes : p.unit_bytes;
    }
  }
  p.tiles_per_img = (p.T + (p.tg ? p.kpos : kTileK) - 1) / (p.tg ? p.kpos : kTileK);
  const long long total = static_cast<long long>(p.imgs) * p.tiles_per_img;
  if (total > 2147483647LL / 4) return false;
  p.total_ktiles = static_cast<int>(total);
  const int sms = sm_count();
  auto n_tiles_of = [&](int acc_n, int n_acc) {
    return p.tg >= 2 ? p.kw * p.upt
           : (p.mode == 0) ? (p.O + acc_n * n_acc - 1) / (acc_n * n_acc) : (p.n_units + n_acc - 1) / n_acc;
  };
  // The K-tiles in splits of four or more: a CTA's time is that of its K-tiles and some five tiles' worth for its
  // start, its partial tile and its share of the reduction.  Next to other streams' calls (SURGEON_SHARE_GPU) the SMs
  // that a layer leaves idle are not idle: splits of eight, and the widest column tiles (320 -> 320 channels of 4096
  // rows take 24 SMs for 23.6 us instead of 144 for 19.5; a Segformer-shaped stack on eight streams 5.0 instead of
  // 5.9 ms, on one stream 8.3 instead of 7.7).
  const int least = share ? 8 : 4;
  const int max_splits = static_cast<int>(std::min<long long>((total + least - 1) / least, 128));
  if (!share && !p.pair && p.tg < 2 && static_cast<long long>(p.m_tiles) * n_tiles_of(p.acc_n, p.n_acc) * max_splits < sms) {
    // The widest column tiles leave SMs without work: narrower ones.  They rebuild the activation once more each, on
    // SMs that would idle, and the partial tile (7 K-tiles' worth at 512 columns: it leaves at 25 to 30 bytes a
    // clock) is written by more of them.
    double best_cost = 1e30;
    int best_n = p.acc_n, best_a = p.n_acc;
    auto consider = [&](int acc_n, int n_acc) {
      const long long tiles = static_cast<long long>(p.m_tiles) * n_tiles_of(acc_n, n_acc);
      const int s = static_cast<int>(std::max<long long>(1, std::min<long long>(max_splits, sms / tiles)));
      const double waves = static_cast<double>((tiles * s + sms - 1) / sms);
      const double cost = waves * ((total + s - 1) / s + 5 + 7.0 * acc_n * n_acc / 512);
      if (cost < best_cost - 1e-9) { best_cost = cost; best_n = acc_n; best_a = n_acc; }
    };
    consider(p.acc_n, p.n_acc);
    if (p.mode == 0) for (int a = 256; a >= 64; a -= 64) { if (a < p.acc_n * p.n_acc) consider(a, 1); }
    else for (int a = p.n_acc - 1; a >= 1; --a) consider(p.acc_n, a);
    p.acc_n = best_n; p.n_acc = best_a;
    if (p.tg) p.b_bytes = p.n_acc * p.unit_bytes;
  }
  if (p.acc_n < 16 || p.acc_n > 256 || p.acc_n % 16 != 0) return false;      // not a shape that an MMA has
  p.n_cols = p.acc_n * p.n_acc;
  p.n_tiles = n_tiles_of(p.acc_n, p.n_acc);
  const long long tiles_mn = static_cast<long long>(p.m_tiles) * p.n_tiles;
  int best = 1;
  double best_cost = 1e30;
  for (int s = 1; s <= max_splits; ++s) {
    const long long ctas = tiles_mn * s;
    const long long waves = (ctas + sms - 1) / sms;
    const int kts = (p.total_ktiles + s - 1) / s;
    const double cost = static_cast<double>(waves) * (kts + 12) + 0.02 * s * tiles_mn / sms;
    if (cost < best_cost - 1e-9) { best_cost = cost; best = s; }
  }
  p.ktiles_per_split = (p.total_ktiles + best - 1) / best;
  p.splits = (p.total_ktiles + p.ktiles_per_split - 1) / p.ktiles_per_split;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.n_cols) p.tmem_cols *= 2;
  if (!size_rings(&p, kStageBytes)) return false;   // the launcher sizes them again for the dtype
  *out = p;
  return true;
}

bool plan_direct(const surgeon_layer_desc& d, bool share, DirectParams* out) {
  struct Tag {};
  return memo_plan<Tag>(d, (use_pairs() ? 1 : 0) + (share ? 2 : 0), out, [&](DirectParams* p) {
    // (a stage of boxes with halo rows can be too large for the rings)
    return compute_plan_direct(d, !use_pairs(), share, p) || compute_plan_direct(d, false, share, p);
  });
}

bool plan_direct_copies(const surgeon_layer_desc& d, DirectParams* out) { return compute_plan_direct(d, false, false, out); }

size_t direct_grad_bf16_bytes(const DirectParams& p) {
  const size_t b = p.tg ? static_cast<size_t>(p.imgs) * p.oh * p.ow * p.o_real * 2
                   : (p.mode == 0) ? static_cast<size_t>(p.T) * p.O * 2
                                 : static_cast<size_t>(p.imgs) * p.copies * p.o_real * p.pitch * 2;
  return (b + 255) & ~static_cast<size_t>(255);
}

// The bf16 copy (or shifted copies) of the output gradient that the tensor maps of the direct
// kernels read: one streaming pre-pass.
cudaError_t launch_direct_prepass(const DirectParams& p, const float* grad_out, void* grad_bf16,
                                  uint32_t* status, cudaStream_t stream) {
  auto run = [&](auto kernel, int grid, long long items) -> cudaError_t {
    note_launches(1);
    return launch_kernel(kernel, dim3(grid), dim3(256), 0, stream, true, grad_out,
                         static_cast<unsigned short*>(grad_bf16), items, p, status);
  };
  cudaError_t e;
  if (p.tg) {
    const long long blocks = static_cast<long long>(p.imgs) * ((p.oh * p.ow + 63) / 64) * ((p.o_real + 63) / 64);
    const long long cap = 8LL * sm_count();
    e = run(grad_transpose_bf16_kernel, static_cast<int>(blocks < cap ? blocks : cap), blocks);
  } else if (p.row_shift) {
    const long long chunks = static_cast<long long>(p.imgs) * p.o_real * (p.pitch >> 3);
    const long long want = (chunks + 255) / 256;
    const long long cap = 32LL * sm_count();
    const int grid = static_cast<int>(want < 1 ? 1 : (want > cap ? cap : want));
    const bool same = (p.kw & 1) && p.pad == (p.kw - 1) / 2 && p.ow == p.in_w &&
                      (reinterpret_cast<uintptr_t>(grad_out) & 15) == 0;
    switch (p.kw) {
      case 2: e = run(grad_cols_bf16_kernel<2, false>, grid, chunks); break;
      case 3:
        if (same) e = run(grad_cols_bf16_kernel<3, true>, grid, chunks);
        else e = run(grad_cols_bf16_kernel<3, false>, grid, chunks);
        break;
      case 5:
        if (same) e = run(grad_cols_bf16_kernel<5, true>, grid, chunks);
        else e = run(grad_cols_bf16_kernel<5, false>, grid, chunks);
        break;
      default:
        if (same) e = run(grad_cols_bf16_kernel<7, true>, grid, chunks);
        else e = run(grad_cols_bf16_kernel<7, false>, grid, chunks);
        break;
    }
  } else if (p.taps > 1) {
    const long long chunks = static_cast<long long>(p.imgs) * p.O * (p.pitch >> 3);
    const long long want = (chunks + 255) / 256;
    const long long cap = 32LL * sm_count();
    const int grid = static_cast<int>(want < 1 ? 1 : (want > cap ? cap : want));
    const bool same = (p.kw & 1) && p.kh == p.kw && p.pad == (p.kw - 1) / 2 && p.ow == p.in_w &&
                      p.oh == p.in_h && (p.kw == 3 || p.kw == 5 || p.kw == 7);
    if (same) {
      const long long items = chunks / p.kw;        // one thread per row shift writes the kw column shifts
      const long long want_s = (items + 255) / 256;
      const int grid_s = static_cast<int>(want_s < 1 ? 1 : (want_s > cap ? cap : want_s));
      if (p.kw == 3) e = run(grad_taps_same_bf16_kernel<3>, grid_s, items);
      else if (p.kw == 5) e = run(grad_taps_same_bf16_kernel<5>, grid_s, items);
      else e = run(grad_taps_same_bf16_kernel<7>, grid_s, items);
    } else {
      e = run(grad_taps_bf16_kernel, grid, chunks);
    }
  } else if (p.mode != 0 && p.pitch != p.T)     // rows padded to a 16-byte pitch for the tensor map
    e = launch_grad_to_bf16_rows(grad_out, static_cast<long long>(p.imgs) * p.O, p.T, p.pitch,
                                 grad_bf16, status, stream);
  else
    e = launch_grad_to_bf16(grad_out, static_cast<long long>(p.imgs) * p.O * p.T, grad_bf16, status, stream);
  return e;
}

// Tensor map over the bf16 gradient copy.  Linear: [T rows][O columns], box 64 columns x 64 rows.
// Conv: [images][copies * O rows][g_len positions], box 64 positions x `box_rows` rows.
cudaError_t encode_direct_grad_map(const DirectParams& p, void* grad_bf16, int box_rows, CUtensorMap* out) {
  CUtensorMap& map = *out;
  const EncodeFn encode = reinterpret_cast<EncodeFn>(tensor_map_encode_fn());
  if (!encode) return cudaErrorNotSupported;
  CUresult r;
  if (p.tg) {
    const cuuint64_t o = static_cast<cuuint64_t>(p.o_real), w = static_cast<cuuint64_t>(p.ow), h = static_cast<cuuint64_t>(p.oh);
    const cuuint64_t dims[4] = {o, w, h, static_cast<cuuint64_t>(p.imgs)};
    const cuuint64_t strides[3] = {o * 2, o * w * 2, o * w * h * 2};
    const cuuint32_t box[4] = {64, static_cast<cuuint32_t>(p.mode == 3 ? p.slot_w : p.in_w),
                               static_cast<cuuint32_t>(p.tg == 2 ? p.map_rows + p.kh - 1 : p.map_rows), 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    r = encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, grad_bf16, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else if (p.mode == 0) {
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(p.O), static_cast<cuuint64_t>(p.T)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(p.O) * 2};
    const cuuint32_t box[2] = {64, static_cast<cuuint32_t>(kTileK)};
    const cuuint32_t estr[2] = {1, 1};
    r = encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, grad_bf16, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  } else {
    const cuuint64_t rows = static_cast<cuuint64_t>(p.copies) * p.o_real;
    const cuuint64_t dims[3] = {static_cast<cuuint64_t>(p.g_len), rows, static_cast<cuuint64_t>(p.imgs)};
    const cuuint64_t strides[2] = {static_cast<cuuint64_t>(p.pitch) * 2,
                                   static_cast<cuuint64_t>(p.pitch) * rows * 2};
    const cuuint32_t box[3] = {static_cast<cuuint32_t>(kTileK),
                               static_cast<cuuint32_t>(box_rows), 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    r = encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, grad_bf16, dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  }
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t launch_direct(const surgeon_compressed& act, const DirectParams& plan,
                          const float* grad_out, void* grad_bf16, float* partial,
                          uint32_t* status, cudaStream_t stream) {
  DirectParams p = plan;
  if (!size_rings(&p, act.dt == 0 && p.mode != 3 ? kStageBytes : 0)) return cudaErrorInvalidValue;
  p.n_words = (act.n + 31) / 32;
  p.few_keep = static_cast<unsigned>(act.n / 8);
  p.n_keep_ptr = reinterpret_cast<const long long*>(reinterpret_cast<const char*>(act.header) +
                                                    offsetof(surgeon_header, n_keep));
  p.partial_blk = (act.n % SURGEON_BLOCK) ? static_cast<unsigned>(act.n / SURGEON_BLOCK) : 0xFFFFFFFFu;
  cudaError_t e = launch_direct_prepass(p, grad_out, grad_bf16, status, stream);
  if (e != cudaSuccess) return e;
  CUtensorMap map;
  e = encode_direct_grad_map(p, grad_bf16, p.pair ? p.acc_n / 2 : p.acc_n, &map);
  if (e != cudaSuccess) return e;
  dim3 grid(p.m_tiles, p.n_tiles, p.splits);
  auto launch = [&](auto kernel) -> cudaError_t {
    cudaError_t err = allow_dynamic_smem(reinterpret_cast<const void*>(kernel), p.smem_bytes);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = static_cast<size_t>(p.smem_bytes);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.pair ? 2 : 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // starts while the gradient pre-pass drains: set-up and the first activation tiles overlap it
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, act.bitmap, act.values, act.block_offsets, map, partial,
                              status, p);
  };
  if (p.mode == 3) {
    // From where on a warp's lanes share each run (70 % / 50 % / 0 % pruned; each lane its own run, and shared: 256 -> 512
    // channels on 56x56, batch 64, fp32 101, 142, 103 and 93, 97, 101 us; 512 -> 1024 on 28x28 79, 112, 126 and 95, 103,
    // 126; bf16 67, 89, 108 and 91, 93, 116, 60 % kept 155 and 101; 1024 -> 2048 on 14x14 54, 67, 77 and 83, 73, 77).
    // Rows that fill two thirds of their slots or less leave a third of the shared lanes without an element: from 55 % kept on (bf16:
    // 1024 -> 2048 on 33x33, batch 22, half pruned 114 us each its own and 207 shared, MODE 2 166; 20 % pruned 222 and 198) or 45 % (fp32:
    // 256 -> 512 on 40x40, batch 61, half pruned 72 and 61); and with up to 64 channels, where half the runs are past the
    // last one as well, never (64 -> 128 on 80x80, batch 61, bf16, 20 % pruned 58 and 77, MODE 2 71).
    const bool padded = 3 * p.ow <= 2 * p.slot_w;
    const int percent = padded ? (p.C <= 64 ? 100 : (act.dt == 0 ? 45 : 55)) : (p.slot_w >= 32 ? 35 : (act.dt == 0 ? 40 : 48));
    p.many_keep = static_cast<unsigned>(act.n * percent / 100);
    e = act.dt ? launch(dw_direct_kernel<1, 3, 0, 1>) : launch(dw_direct_kernel<0, 3, 0, 1>);
    note_launches(1);
    return e;
  }
  if (p.tg) {
    switch (p.tg * 2 + (act.dt ? 1 : 0)) {
      case 2: e = launch(dw_direct_kernel<0, 1, 0, 1>); break;
      case 3: e = launch(dw_direct_kernel<1, 1, 0, 1>); break;
      case 4: e = launch(dw_direct_kernel<0, 1, 0, 2>); break;
      case 5: e = launch(dw_direct_kernel<1, 1, 0, 2>); break;
      case 6: e = launch(dw_direct_kernel<0, 1, 0, 3>); break;
      case 7: e = launch(dw_direct_kernel<1, 1, 0, 3>); break;
      case 8: e = launch(dw_direct_kernel<0, 1, 0, 4>); break;
      case 9: e = launch(dw_direct_kernel<1, 1, 0, 4>); break;
      case 10: e = launch(dw_direct_kernel<0, 1, 0, 5>); break;
      default: e = launch(dw_direct_kernel<1, 1, 0, 5>); break;
    }
    note_launches(1);
    return e;
  }
  const int key = p.mode * 4 + (act.dt ? 2 : 0) + p.pair;
  switch (key) {
    case 0: e = launch(dw_direct_kernel<0, 0, 0>); break;
    case 1: e = launch(dw_direct_kernel<0, 0, 1>); break;
    case 2: e = launch(dw_direct_kernel<1, 0, 0>); break;
    case 3: e = launch(dw_direct_kernel<1, 0, 1>); break;
    case 4: e = launch(dw_direct_kernel<0, 1, 0>); break;
    case 5: e = launch(dw_direct_kernel<0, 1, 1>); break;
    case 6: e = launch(dw_direct_kernel<1, 1, 0>); break;
    case 7: e = launch(dw_direct_kernel<1, 1, 1>); break;
    case 8: e = launch(dw_direct_kernel<0, 2, 0>); break;
    case 9: e = launch(dw_direct_kernel<0, 2, 1>); break;
    case 10: e = launch(dw_direct_kernel<1, 2, 0>); break;
    default: e = launch(dw_direct_kernel<1, 2, 1>); break;
  }
  note_launches(1);
  return e;
}

}  // namespace surgeon
