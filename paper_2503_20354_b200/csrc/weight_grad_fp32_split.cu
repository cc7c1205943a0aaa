// fp32 path of surgeon_weight_grad on the tensor cores (Algorithm 1: Reshape and gradient steps, Eq. 2).
//
// An fp32 number is the sum of three bf16 numbers, exactly: x1 = bf16(x), x2 = bf16(x - x1), x3 = x - x1 - x2 (24
// significant bits in 3 x 8, both differences exact).  A product is then the sum of nine products of bf16 numbers, each
// exact in fp32; six of them are formed (x1 y1, x1 y2, x2 y1, x2 y2, x1 y3, x3 y1), the other three are 2^-26 of it and
// less.  For bf16 activations x = x1, and three products are all.  Both operands are first multiplied by 2^24 (exact), which
// the reduction takes out: without it numbers below 2^-109 lost their low parts, however large others were (an output channel
// of 1e-36 beside ordinary ones: 3e-5 of its row of dW, one of 1e-40 a quarter of it; now 1e-7).
//
// The tensor cores add with truncation, so no long chain of large terms runs in them: x1 y1 is summed over one K-tile of 64
// positions, from zero, and leaves for fp32 registers, where it is added rounding to nearest.  The small products have an
// accumulator of their own, 2^-9 of the whole (and so is what is cut off it), which is added at the end of the chunk.  A
// chunk of at most 32 K-tiles (2048 terms) is a partial sum, and the partial sums are added in double in a fixed order.
// Error against 64 bits (320 -> 320 channels, 3x3 on 16x16, batch 16; relative 2-norm; the CUDA-core kernel's in brackets): nothing
// pruned 1.0e-7 (3.4e-7), 90 % pruned 5.8e-8 (1.6e-7), 99 % 3.8e-8 (6.1e-8).  (With the small products first in the
// same accumulator it was 1.1e-7, 1.05e-7 and more than before from 97 % on: every sum was cut off toward zero.)
// 13 layers of all kinds, both types, seven pruning ratios, 182 calls: the 2-norm of the error is 0.49 of the CUDA cores' in the
// geometric mean and above it in none.  Part of it has one sign, since what is cut off is cut off toward zero: unpruned, dW is 2.3e-8
// to 6.1e-8 of itself too small, half pruned 0.8e-8 to 2.8e-8, from 70 % on within 6e-9 (CUDA cores: within 9e-9 at all ratios).  The
// largest error of one element is above the CUDA cores' in 13 calls, most of them pruned by 97 % and more, by up to 1.22.
//
//   dW[m, nn] = sum_k G[k, m] * Acol[k, nn],  nn = (c, r, s) -> MMA M (128), m = output channel -> MMA N (up to 160),
//   k = (b, y, x) over all images, or the row t of a linear layer -> MMA K, 64 per stage.
//
// 16 warps rebuild the activation tile from the store (a lane owns 16 positions of one column, or 16 channels of one
// row) and cut it into its planes, and after each K-tile take the sums of the one before out of tensor memory: two stages
// of shared memory, two accumulators of the large products.  A tile's values are under way while the sums are taken, and the
// words of the one after it.  A pre-pass writes the gradient's planes as they lie in shared memory: one bulk copy a tile.
//
// Measured on 320 -> 320 channels, 3x3 on 16x16, batch 16 (7.5 GFLOP): 264 us on CUDA cores, 66-71 now, of which the pre-pass
// takes 4, this kernel 55 and the reduction 4.  70 % pruned, a K-tile takes 4000 clocks (start and epilogue included), its MMAs
// 1920 at their nominal rate; tensor pipe 46 %, issue slots 64 %, DRAM 2 % busy: the warps' instructions and what they wait for are the bound.
// (Clock stamps in a copy of the kernel: store 750, asking for values 1300, sums 800, or 2000 beside MMAs.)  MMAs issued by the
// warps in turn instead of by a warp of their own took 1.6 times as long, since whoever issues is late for the next tile.
//
// Infinities and NaN, operands from 2^104 on and calls whose largest operands multiply to 2^64 and more (which the
// factor could make infinite) are seen from the largest magnitudes, which every block records; a wait that ran out
// records one too.  The CUDA-core kernel then computes the whole call again.
#include <cuda.h>

#include <algorithm>

#include "fp32_path.cuh"
#include "tc_common.cuh"
#include "weight_grad_tc_conv.cuh"

namespace surgeon {

namespace {

using namespace tc;

constexpr int kTileM = 128, kTileK = kSplitTileK;
// 16 warps work, one issues MMAs, one loads.  Five warpgroups are launched with 96 registers a thread; the last one gives
// up 72 of them and the others take 16 more: 512 x 112 + 128 x 24 <= 640 x 96.
constexpr int kWarps = 16, kThreads = 32 * (kWarps + 4);
constexpr int kRegsWork = 112, kRegsIssue = 24;
static_assert(32 * kWarps * kRegsWork + 128 * kRegsIssue <= kThreads * 96, "registers of the launch");
constexpr int kMaxTileN = 160;                   // 40 sums a thread; two accumulators in 512 columns
constexpr int kPlaneA = kTileM * kTileK * 2;     // 16 KB
constexpr int kMaxTiles = 2048 / kTileK;         // K-tiles of one chunk at most
// The planes take 1.5 times the gradient (more where columns are padded), so a large layer is done in slabs: as many chunks at
// a time as 128 MB of planes hold, or half the fp32 gradient where that is more (what the bf16 path's copy of it takes).
// 64 -> 256 channels 1x1 on 56x56, batch 64: 318 MB of scratch and 200 us in one piece, 117 and 218 in three slabs (8 MB of them
// partial sums); with 64 MB at most it would be 97 and 228.  3x3, 160 -> 160 on 32x32, batch 200: 303 MB and 708 us, 172 and 739.
constexpr long long kMaxPlanes = 128LL << 20;
constexpr double kSlabCost = 4.0;                // of a further slab, in K-tiles
constexpr int kLeastTiles = 20;                  // chunks of fewer K-tiles only while the partial sums are below
constexpr double kMaxPartials = 32 << 20;
constexpr float kSplitScale = static_cast<float>(1 << kSplitShift);

// x0, x1 times 2^kSplitShift -> their three parts, two to a word.  (Multiplied before the first rounding: a subnormal number's first
// part has fewer bits, and the products that are left out would be up to 2^-17 of the whole.)
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& p1, uint32_t& p2, uint32_t& p3) {
  x0 *= kSplitScale;
  x1 *= kSplitScale;
  p1 = pack_bf16x2(x0, x1);
  x0 -= __uint_as_float(p1 << 16);
  x1 -= __uint_as_float(p1 & 0xFFFF0000u);
  p2 = pack_bf16x2(x0, x1);
  x0 -= __uint_as_float(p2 << 16);
  x1 -= __uint_as_float(p2 & 0xFFFF0000u);
  p3 = pack_bf16x2(x0, x1);
}
// Two bf16 numbers times 2^kSplitShift.
__device__ __forceinline__ uint32_t scale_bf16x2(uint32_t x) {
  uint32_t r;
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(static_cast<uint32_t>((127 + kSplitShift) << 7) * 0x10001u));
  return r;
}
// The packed value `idx` into r where `on`.
template <int DT>
__device__ __forceinline__ void take_packed(uint32_t& r, const void* __restrict__ values, uint32_t idx, bool on) {
  const unsigned char* src = reinterpret_cast<const unsigned char*>(values) + static_cast<size_t>(idx) * (DT == 0 ? 4 : 2);
  if (DT == 0)
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.u32 %0, [%1];\n\t}"
                 : "+r"(r) : "l"(src), "r"(static_cast<uint32_t>(on)));
  else
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\t@q ld.global.nc.u16 %0, [%1];\n\t}"
                 : "+r"(r) : "l"(src), "r"(static_cast<uint32_t>(on)));
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr) : "memory");
}
// (the registers pass through it, so that nothing uses them before)
__device__ __forceinline__ void tmem_ld8_wait(uint32_t (&r)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :: "memory");
}
// MN-major operand, 128-byte swizzle: rows of 64 elements per k, the next 64 along M or N a slab of 64 k-rows on.
__device__ __forceinline__ uint64_t make_desc_mn64(uint32_t saddr) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) | static_cast<uint64_t>((kTileK * 128) >> 4) << 16 |
         static_cast<uint64_t>(1024 >> 4) << 32 | static_cast<uint64_t>(1) << 46 | static_cast<uint64_t>(2) << 61;
}

// The planes of a slab of the gradient, cut into the pieces that a CTA loads for a K-tile, byte for byte as they lie in its
// shared memory: [K-tile][column tile][plane][tile_n x 64].  Eight columns a thread.  `most`: a word per block.
__global__ void __launch_bounds__(256)
grad_split_kernel(const float* __restrict__ grad, unsigned char* __restrict__ out, uint32_t* __restrict__ most, SplitGeom g) {
  pdl_wait();
  pdl_trigger();
  // a row is an output channel, its columns the positions of all images (linear: a row t, its columns channels)
  const int n_rows = g.linear ? g.K : g.O, n_cols = g.linear ? g.O : g.K;
  const int k0 = g.kt0 * kTileK, k_here = slab_tiles(g) * kTileK;
  const int rows = g.linear ? k_here : g.nt * g.tile_n, per_row = (g.linear ? g.nt * g.tile_n : k_here) >> 3;
  const long long items = static_cast<long long>(rows) * per_row;
  const size_t plane = static_cast<size_t>(g.tile_n) * kTileK * 2;
  uint32_t largest = 0;
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < items;
       i += static_cast<long long>(gridDim.x) * blockDim.x) {
    int row = static_cast<int>(i / per_row), col = static_cast<int>(i - static_cast<long long>(row) * per_row) * 8;
    if (g.linear) row += k0;
    else col += k0;
    // a row's columns are in pieces of P, one per image (linear: in one piece)
    const uint32_t img = g.linear ? 0u : divide(col, g.by_p), p = col - img * g.P;
    const float* at = grad + (g.linear ? static_cast<size_t>(row) * g.O + col : (static_cast<size_t>(img) * g.O + row) * g.P + p);
    const size_t skip = g.linear ? 0 : static_cast<size_t>(g.O - 1) * g.P;        // from an image's end to the next one
    const int len = row < n_rows ? n_cols : 0;
    float x[8];
    uint32_t q = p;
    if (g.vec) {                                 // (four columns from a multiple of 4 on are 16 bytes of one piece)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 v = col + 4 * h < len ? __ldg(reinterpret_cast<const float4*>(at)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        x[4 * h] = v.x; x[4 * h + 1] = v.y; x[4 * h + 2] = v.z; x[4 * h + 3] = v.w;
        at += 4;
        q += 4;
        if (!g.linear && q == static_cast<uint32_t>(g.P)) { q = 0; at += skip; }
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        x[e] = col + e < len ? __ldg(at) : 0.0f;
        ++at;
        if (!g.linear && ++q == static_cast<uint32_t>(g.P)) { q = 0; at += skip; }
      }
    }
    uint32_t a[4], b[4], c[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      split2(x[2 * e], x[2 * e + 1], a[e], b[e], c[e]);
      largest = __vmaxu2(largest, a[e] & 0x7FFF7FFFu);
    }
    const int o = g.linear ? col : row, k = (g.linear ? row : col) - k0, j = o / g.tile_n, n = o - j * g.tile_n;
    const size_t place = (static_cast<size_t>(k / kTileK) * g.nt + j) * 3 * plane +
                         (g.linear ? (n >> 6) * (kTileK * 128) + tile_off(k % kTileK, (n & 63) >> 3) : tile_off(n, (k % kTileK) >> 3));
    if (!SURGEON_IN_BOUNDS(place + 2 * plane + 15, split_planes_bytes(g), g.status)) continue;
    unsigned char* to = out + place;
    *reinterpret_cast<uint4*>(to) = make_uint4(a[0], a[1], a[2], a[3]);
    *reinterpret_cast<uint4*>(to + plane) = make_uint4(b[0], b[1], b[2], b[3]);
    *reinterpret_cast<uint4*>(to + 2 * plane) = make_uint4(c[0], c[1], c[2], c[3]);
  }
  __shared__ uint32_t s_most;
  if (threadIdx.x == 0) s_most = 0;
  __syncthreads();
  largest = __reduce_max_sync(0xFFFFFFFFu, max(largest & 0xFFFFu, largest >> 16));
  if (lane_id() == 0) atomicMax(&s_most, largest);
  __syncthreads();
  if (threadIdx.x == 0) most[blockIdx.x] = s_most;
}

// KIND: 0 linear (both operands MN-major), 1 convolution of stride one (K-major), 2 of another stride.
template <int DT, int KIND>
__global__ void __launch_bounds__(kThreads, 1)
dw_split_kernel(const uint32_t* __restrict__ bitmap, const void* __restrict__ values,
                const uint32_t* __restrict__ offsets, const unsigned char* __restrict__ planes,
                float* __restrict__ partial, uint32_t* __restrict__ most, SplitGeom g) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  constexpr int NA = DT == 0 ? 3 : 1;            // planes of the activation
  const int plane_b = g.tile_n * kTileK * 2, stage_bytes = NA * kPlaneA + 3 * plane_b;
  __shared__ __align__(8) unsigned long long bars[6];
  __shared__ uint32_t tmem_slot, s_most;
  __shared__ volatile uint32_t fail;

  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t lane = lane_id();
  const int n0 = blockIdx.x * kTileM, o0 = blockIdx.y * g.tile_n;
  const int chunk = g.chunk0 + static_cast<int>(blockIdx.z), kt_begin = chunk * g.per_chunk, n_kt = min(g.per_chunk, g.k_tiles - kt_begin);
  const uint32_t full_a = smem_u32(bars), full_b = smem_u32(bars + 2), done = smem_u32(bars + 4);
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(full_a + 8 * s, kWarps);
      mbar_init(full_b + 8 * s, 1);
      mbar_init(done + 8 * s, 1);
    }
    fail = 0;
    s_most = 0;
    fence_barrier_init();
  }
  if (warp == kWarps) tmem_alloc(smem_u32(&tmem_slot), g.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  pdl_trigger();                                 // (the store was there before the pre-pass began)

  if (warp >= kWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsIssue));
    if (warp == kWarps && lane == 0) {
      // ================= MMA issuer =================
      constexpr uint64_t kStep = KIND == 0 ? 128 : 2;
      constexpr int kProducts = DT == 0 ? 6 : 3;
      constexpr int pa[6] = {0, 0, 1, 1, 0, 2}, pb[6] = {0, 1, 0, 1, 2, 0};          // the large one first
      const uint32_t idesc = make_idesc(kTileM, g.tile_n) | (KIND == 0 ? ((1u << 15) | (1u << 16)) : 0u);
      for (int it = 0; it < n_kt; ++it) {
        const int s = it & 1;
        const uint32_t parity = (it >> 1) & 1;
        if (fail || !mbar_wait_suspend(full_b + 8 * s, parity) || !mbar_wait_suspend(full_a + 8 * s, parity)) {
          fail = 1;                              // (the MMAs under way write to tensor memory)
          if (it > 0) mbar_wait_suspend(done + 8 * (s ^ 1), ((it - 1) >> 1) & 1);
          break;
        }
        tc_fence_after();
        const uint32_t at = smem_u32(smem) + s * stage_bytes;
        const uint64_t da = KIND == 0 ? make_desc_mn64(at) : make_desc(at);
        const uint64_t db = KIND == 0 ? make_desc_mn64(at + NA * kPlaneA) : make_desc(at + NA * kPlaneA);
#pragma unroll
        for (int i = 0; i < kProducts; ++i) {
          const int x = DT == 0 ? pa[i] : 0, y = DT == 0 ? pb[i] : i;
          const uint64_t dx = da + static_cast<uint64_t>(x * (kPlaneA >> 4)), dy = db + static_cast<uint64_t>(y * (plane_b >> 4));
          const uint32_t to = tmem_base + (i == 0 ? s : 2) * g.tile_n, fresh = i == 0 || (i == 1 && it == 0) ? 1u : 0u;
#pragma unroll
          for (uint64_t kk = 0; kk < 4; ++kk) umma_bf16(to, dx + kk * kStep, dy + kk * kStep, idesc, kk > 0 ? 1u : fresh ^ 1u);
        }
        umma_commit(done + 8 * s);
      }
    } else if (warp == kWarps + 1 && lane == 0) {
      // ================= the gradient's planes =================
      pdl_wait();                                // they are written
      int it = 0;
      for (; it < n_kt; ++it) {
        const int s = it & 1;
        if (it >= 2 && (fail || !mbar_wait_suspend(done + 8 * s, ((it - 2) >> 1) & 1))) { fail = 1; break; }
        mbar_arrive_expect_tx(full_b + 8 * s, 3u * plane_b);
        bulk_load(smem_u32(smem) + s * stage_bytes + NA * kPlaneA,
                  planes + (static_cast<size_t>(kt_begin - g.kt0 + it) * gridDim.y + blockIdx.y) * (3u * plane_b), 3u * plane_b, full_b + 8 * s);
      }
      // (the loads under way write to shared memory)
      for (int i = max(0, it - 2); i < it; ++i) mbar_wait_suspend(full_b + 8 * (i & 1), (i >> 1) & 1);
    }
    __syncwarp();
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsWork));
    // ================= a tile of the activation, then the sums of the tile before =================
    float acc[5][8];
#pragma unroll
    for (int u = 0; u < 5; ++u)
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[u][i] = 0.0f;
    const int col0 = (warp >> 2) * g.warp_cols;  // this warp's columns of the accumulator, and how many there are
    const int n_cols = min(g.warp_cols, g.tile_n - col0);
    uint32_t largest = 0;
    // convolution: this lane's column (c, r, s) and which 16 positions of the tile; linear: row and 16 channels
    const int row = KIND == 0 ? 4 * warp + static_cast<int>(lane >> 3) : 8 * warp + static_cast<int>(lane >> 2);
    const int part = KIND == 0 ? lane & 7 : lane & 3;
    int c = 0, ry = 0, rx = 0, n_ch = 0;         // (ry, rx: input row and column of output position (0, 0))
    if (KIND == 0) {
      c = n0 + 16 * part;
      n_ch = max(0, min(16, g.C - c));
    } else {
      const int nn = n0 + row;
      n_ch = nn < g.N ? 16 : 0;
      c = nn / g.RS;
      const int rs = nn - c * g.RS;
      ry = rs / g.KW;
      rx = rs - ry * g.KW - g.pad;
      ry -= g.pad;
    }
    // A piece: positions of one output row inside the map, at most 32 input elements wide (linear: the channels).  Its
    // words are asked for when it is made, and used when its values are asked for.
    uint32_t j = 0, base = 0, next = 0;          // its first element, the kept ones before that's block, the word after the block
    uint4 q = make_uint4(0, 0, 0, 0);            // the block's words
    int e0 = 0, n = 0;                           // its first element of the lane's 16, and how many
    int img = 0, y = 0, x = 0, kp = 0;           // (convolution) the lane's first position of the tile that is asked for
    if (KIND != 0) {
      kp = kt_begin * kTileK + 16 * part;
      img = divide(kp, g.by_p);
      const int p = kp - img * g.P;
      y = divide(p, g.by_ow);
      x = p - y * g.OW;
    }
    auto fetch = [&]() {
      const uint32_t blk = j >> kBlockShift, w0 = blk * kBlockWords;
      base = __ldg(offsets + blk);
      next = 0;
      if (w0 + 4 <= g.n_words) {
        q = __ldg(reinterpret_cast<const uint4*>(bitmap) + blk);
      } else {                                   // the last, partial block
        q.x = __ldg(bitmap + w0);
        q.y = w0 + 1 < g.n_words ? __ldg(bitmap + w0 + 1) : 0u;
        q.z = w0 + 2 < g.n_words ? __ldg(bitmap + w0 + 2) : 0u;
      }
      if ((j & 127u) > 96u && w0 + 4 < g.n_words) next = __ldg(bitmap + w0 + 4);
    };
    // the piece from position `at` of the lane's n_e on, at (im, yy, xx); returns how many positions it covers
    auto make = [&](int at, int n_e, int im, int yy, int xx) -> int {
      int len = min(n_e - at, g.OW - xx), ix = xx * g.stride + rx, skip = 0;         // skip: positions left of the map
      if (KIND == 2) len = min(len, g.most_len);
      const int iy = yy * g.stride + ry;
      if (ix < 0) { skip = KIND == 1 ? -ix : (-ix + g.stride - 1) / g.stride; ix += skip * g.stride; }
      const int right = g.W - 1 - ix;
      e0 = at + skip;
      n = min(len - skip, (KIND == 1 ? right : (right < 0 ? -1 : right / g.stride)) + 1);
      if (static_cast<uint32_t>(iy) >= static_cast<uint32_t>(g.H)) n = 0;
      j = ((im * g.C + c) * g.H + iy) * g.W + ix;
      if (n > 0) fetch();
      return len;
    };
    int n_e = 0, covered = 0;                    // the lane's elements of the tile that is asked for; up to the piece's end
    auto first = [&](int it) {                   // the first piece of tile `it`, the tiles in order
      n = 0;
      n_e = covered = 0;
      if (KIND == 0) {
        const int t = (kt_begin + it) * kTileK + row;
        if (n_ch > 0 && t < g.K) {
          n = n_ch;
          j = static_cast<uint32_t>(t) * g.C + c;
          fetch();
        }
      } else {
        n_e = min(16, g.K - kp);
        if (n_ch > 0 && n_e > 0) covered = make(0, n_e, img, y, x);
        else n_e = 0;
      }
    };
    auto advance = [&]() {                       // 64 positions on
      kp += kTileK;
      x += g.step_x;
      y += g.step_y;
      if (x >= g.OW) { x -= g.OW; ++y; }
#pragma unroll 1
      while (y >= g.OH) { y -= g.OH; ++img; }
    };
    uint32_t v[16];
    auto values_of_piece = [&]() {
      if (n <= 0) return;
      const uint32_t wq = (j >> 5) & 3u, sh = j & 31u;
      const uint32_t w0 = wq == 0 ? q.x : (wq == 1 ? q.y : (wq == 2 ? q.z : q.w));
      const uint32_t w1 = wq == 3 ? next : (wq == 0 ? q.y : (wq == 1 ? q.z : q.w));
      uint32_t idx = base + (wq > 0 ? __popc(q.x) : 0) + (wq > 1 ? __popc(q.y) : 0) + (wq > 2 ? __popc(q.z) : 0) +
                     __popc(w0 & ((1u << sh) - 1u));
      const uint32_t win = __funnelshift_r(w0, w1, sh);
      if (KIND != 2) {
        const uint32_t m = (win & ((1u << n) - 1u)) << e0;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          take_packed<DT>(v[e], values, idx, m & (1u << e));
          if (m & (1u << e)) ++idx;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int at = (e - e0) * g.stride;    // its bit of the window
          const bool in = e >= e0 && e < e0 + n;
          const uint32_t below = in ? (1u << at) - 1u : 0u;
          take_packed<DT>(v[e], values, idx + __popc(win & below), in && ((win >> (at & 31)) & 1u));
        }
      }
    };
    auto ask = [&](int it) {                     // for the values of tile `it`, whose first piece is made; then for the next one's words
#pragma unroll
      for (int e = 0; e < 16; ++e) v[e] = 0u;
      values_of_piece();
      if (KIND != 0) {
        if (covered < n_e) {
          int im = img, yy = y, xx = x, last = covered;
#pragma unroll 1
          for (;;) {
            xx += last;
            if (xx >= g.OW) {
              xx = 0;
              if (++yy == g.OH) { yy = 0; ++im; }
            }
            if (covered >= n_e) break;
            last = make(covered, n_e, im, yy, xx);
            covered += last;
            values_of_piece();
          }
        }
        advance();
      }
      if (it + 1 < n_kt) first(it + 1);
    };
    auto add_sums = [&](int which) {             // this warp's part of an accumulator
      const uint32_t at = tmem_base + which * g.tile_n + (static_cast<uint32_t>((warp & 3) * 32) << 16) + col0;
#pragma unroll
      for (int u0 = 0; u0 < 5; u0 += 2) {
        uint32_t d[2][8];
#pragma unroll
        for (int u = 0; u < 2; ++u)
          if (u0 + u < 5 && 8 * (u0 + u) < n_cols) tmem_ld8(at + 8 * (u0 + u), d[u]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          if (u0 + u < 5 && 8 * (u0 + u) < n_cols) {
            tmem_ld8_wait(d[u]);
#pragma unroll
            for (int i = 0; i < 8; ++i) acc[(u0 + u) % 5][i] += __uint_as_float(d[u][i]);
          }
        }
      }
    };
    first(0);
    ask(0);
    for (int it = 0; it <= n_kt; ++it) {
      if (it < n_kt) {
        // ---- the values in planes ----
        unsigned char* stage = smem + (it & 1) * stage_bytes;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          unsigned char* dst = stage + (KIND == 0 ? (part >> 2) * (kTileK * 128) + tile_off(row, 2 * (part & 3) + h)
                                                  : tile_off(row, 2 * part + h));
          uint32_t w[3][4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint32_t x0 = v[8 * h + 2 * e], x1 = v[8 * h + 2 * e + 1];
            if (DT == 0) split2(__uint_as_float(x0), __uint_as_float(x1), w[0][e], w[1][e], w[2][e]);
            else w[0][e] = scale_bf16x2(x0 | (x1 << 16));
            largest = __vmaxu2(largest, w[0][e] & 0x7FFF7FFFu);
          }
#pragma unroll
          for (int i = 0; i < NA; ++i)
            *reinterpret_cast<uint4*>(dst + i * kPlaneA) = make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(full_a + 8 * (it & 1));
        if (it + 1 < n_kt) ask(it + 1);
      }
      if (it > 0) {
        // ---- the sums of the tile before ----
        const int s = (it - 1) & 1;
        const bool ok = !fail && mbar_wait_suspend(done + 8 * s, ((it - 1) >> 1) & 1);
        if (!__all_sync(0xFFFFFFFFu, ok)) { fail = 1; break; }
        tc_fence_after();
        add_sums(s);
        tc_fence_before();                       // (the next tile's arrival frees this accumulator)
      }
    }
    if (__all_sync(0xFFFFFFFFu, fail == 0)) add_sums(2);       // the small products
    largest = __reduce_max_sync(0xFFFFFFFFu, max(largest & 0xFFFFu, largest >> 16));
    if (lane == 0) atomicMax(&s_most, largest);
    // ---- the partial sums ----
    const int nn = n0 + 32 * (warp & 3) + static_cast<int>(lane);
    float* out = partial + static_cast<size_t>(chunk) * g.O * g.N;
    if (nn < g.N) {
#pragma unroll
      for (int u = 0; u < 5; ++u) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int o = o0 + col0 + 8 * u + i;
          if (8 * u + i < n_cols && o < g.O &&
              SURGEON_IN_BOUNDS((static_cast<size_t>(chunk) * g.O + o) * g.N + nn, static_cast<size_t>(g.chunks) * g.O * g.N, g.status))
            out[static_cast<size_t>(o) * g.N + nn] = acc[u][i];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWarps) tmem_dealloc(tmem_base, g.tmem_cols);
  const int cta = (chunk * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (tid == 0 && SURGEON_IN_BOUNDS(cta, g.ctas, g.status)) most[cta] = fail ? 0xFFFFu : s_most;
}

bool compute_plan_split(const surgeon_layer_desc& d, SplitGeom* out) {
  SplitGeom g{};
  const long long rows = d.batch;
  const int OH = (d.h + 2 * d.pad - d.kh) / d.stride + 1, OW = (d.w + 2 * d.pad - d.kw) / d.stride + 1;
  const long long P = d.kind == 1 ? static_cast<long long>(OH) * OW : 1, K = rows * P;
  const long long N = static_cast<long long>(d.c_in) * d.kh * d.kw;
  if (K < 1 || K > (1LL << 30) || N > (1LL << 30) || d.c_out > (1 << 30)) return false;
  // Rows of fewer than four positions: a rank computation for each piece costs more than the products save.
  if (d.kind == 1 && (OW < 4 || d.stride > 8)) return false;
  // Linear layers of up to 16 rows: a quarter of a K-tile at most, and the CUDA cores launch two kernels less.  Time here over
  // time there, fp32 and bf16, in replays of a graph: 1-4 rows 1.77 and 1.56 (10 instead of 5.6 us for 10 to 3072 outputs), 5-8 rows 1.64
  // and 1.35, 9-16 rows 1.31 and 1.05; 17-23 rows 1.10 and 0.85, 24-32 rows 0.95 and 0.69.
  if (d.kind != 1 && d.batch <= 16) return false;
  // A small layer of stride 2 takes as long on the CUDA cores, which start sooner (0.06 GFLOP, fp32: 64 -> 64 channels,
  // 3x3 on 56x56 13.3 us and here 14.6, 256 -> 256 on 14x14 14.4 and 15.2; 0.15 GFLOP 14.9 and 13.9).
  if (d.stride > 1 && 2.0 * static_cast<double>(K) * d.c_out * static_cast<double>(N) < 1e8) return false;
  // Strides of 7 and 8: pieces of five and four positions, a rank computation each.  With more than 64 outputs the CUDA
  // cores rebuild them for every 64 (0.42-0.9 of their time here), with few inputs they lack columns (3-8: 0.76-1.0, 16-32: 0.96-1.05); else
  // they are the faster ones: 64-128 inputs, 16-64 outputs, 0.1-4 GFLOP 1.02-1.19 of their time here in the mean, 1.48 at most
  // (64 -> 64, 8x8 stride 8 on 56x56, batch 16, fp32: 33 us there, 44 here).  Strides 5 and 6: 0.97-1.0.
  if (d.kind == 1 && d.stride >= 7 && d.c_out <= 64 && d.c_in >= 64) return false;
  g.C = d.c_in; g.H = d.h; g.W = d.w; g.O = d.c_out; g.KW = d.kw; g.RS = d.kh * d.kw;
  g.stride = d.stride; g.pad = d.pad; g.OH = OH; g.OW = OW;
  g.P = static_cast<int>(P); g.K = static_cast<int>(K); g.N = static_cast<int>(N);
  g.most_len = 31 / d.stride + 1;
  g.step_y = d.kind == 1 ? kTileK / OW : 0;
  g.step_x = d.kind == 1 ? kTileK % OW : 0;
  g.linear = d.kind == 1 ? 0 : 1;
  g.vec = (g.linear ? d.c_out % 4 == 0 : P % 4 == 0) ? 1 : 0;
  g.n_words = static_cast<uint32_t>((rows * d.c_in * d.h * d.w + 31) / 32);
  g.by_p = make_div(g.P);
  g.by_ow = make_div(d.kind == 1 ? g.OW : 1);
  // Columns: as few tiles as 160 allows, of equal width (linear: slabs of 64).
  if (d.kind == 1) {
    g.nt = (g.O + kMaxTileN - 1) / kMaxTileN;
    g.tile_n = ((g.O + g.nt - 1) / g.nt + 15) / 16 * 16;
  } else {
    g.tile_n = g.O <= 64 ? 64 : 128;
  }
  g.nt = (g.O + g.tile_n - 1) / g.tile_n;
  g.mt = (g.N + kTileM - 1) / kTileM;
  if (g.nt > 65535) return false;
  g.warp_cols = (g.tile_n + 31) / 32 * 8;
  g.tmem_cols = 32;
  while (g.tmem_cols < 3 * g.tile_n) g.tmem_cols *= 2;
  g.k_tiles = (g.K + kTileK - 1) / kTileK;
  // K-tiles per chunk and chunks per slab: as many rounds of CTAs (one per SM) as it takes, each as short as possible; a
  // chunk costs about three K-tiles (start, epilogue, its part of the reduction) on top of its own, a slab kSlabCost.
  const long long tiles = static_cast<long long>(g.mt) * g.nt;
  const long long room = std::max<long long>(std::max<long long>(kMaxPlanes, 2 * K * d.c_out) / (static_cast<long long>(g.nt) * 3 * g.tile_n * kTileK * 2), kMaxTiles);
  const int sms = sm_count();
  const double chunk_cost = 0.6e-6 * g.O * g.N;  // written and read again, in K-tiles
  double best = 1e300;
  for (int per = 1; per <= kMaxTiles; ++per) {
    const long long chunks = (g.k_tiles + per - 1) / per;
    if (chunks > 65535) continue;                // (blockIdx.z)
    const long long least = (chunks + room / per - 1) / (room / per);
    if (least > 1 && per < kLeastTiles && 4.0 * chunks * g.O * g.N > kMaxPartials) continue;
    for (long long slabs = least; slabs <= (least == 1 ? 1 : least + 3) && slabs <= chunks; ++slabs) {
      const long long each = (chunks + slabs - 1) / slabs, last = chunks - (slabs - 1) * each;
      if (last < 1) continue;
      const double cost = static_cast<double>((slabs - 1) * ((tiles * each + sms - 1) / sms) + (tiles * last + sms - 1) / sms) * (per + 3.0) +
                          (slabs > 1 ? kSlabCost * (slabs - 1) + chunk_cost * chunks : 0.0);
      if (cost <= best) { best = cost; g.per_chunk = per; g.slabs = static_cast<int>(slabs); g.slab_chunks = static_cast<int>(each); }
    }
  }
  if (!g.per_chunk) return false;
  g.chunks = (g.k_tiles + g.per_chunk - 1) / g.per_chunk;
  if (tiles * g.chunks > (1LL << 30)) return false;
  g.ctas = static_cast<int>(tiles * g.chunks);
  const long long items = static_cast<long long>(slab_tiles(g)) * kTileK * g.nt * g.tile_n / 8;
  g.grad_blocks = static_cast<int>(std::min<long long>((items + 255) / 256, 4LL * sms));
  *out = g;
  return true;
}

}  // namespace

bool plan_split(const surgeon_layer_desc& d, SplitGeom* out) {
  struct Tag {};
  return memo_plan<Tag>(d, 0, out, [&](SplitGeom* g) { return compute_plan_split(d, g); });
}

cudaError_t launch_split(const surgeon_compressed& act, const SplitGeom& plan, const float* grad_out, void* planes,
                         float* partial, uint32_t* most, cudaStream_t stream) {
  SplitGeom g = plan;
  g.status = &act.header->status;
  const int smem = 2 * ((act.dt == 0 ? 3 : 1) * kPlaneA + 3 * g.tile_n * kTileK * 2) + 1024;
  auto launch = [&](auto kernel) -> cudaError_t {
    cudaError_t e = allow_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
    for (int slab = 0; slab < g.slabs && e == cudaSuccess; ++slab) {
      g.chunk0 = slab * g.slab_chunks;
      g.kt0 = g.chunk0 * g.per_chunk;
      const int chunks = std::min(g.slab_chunks, g.chunks - g.chunk0);
      e = launch_kernel(grad_split_kernel, dim3(g.grad_blocks), dim3(256), 0, stream, true, grad_out,
                        static_cast<unsigned char*>(planes), most + slab * g.grad_blocks, g);
      if (e != cudaSuccess) break;
      e = launch_kernel(kernel, dim3(g.mt, g.nt, chunks), dim3(kThreads), smem, stream, true, act.bitmap,
                        static_cast<const void*>(act.values), act.block_offsets, static_cast<const unsigned char*>(planes),
                        partial, most + g.slabs * g.grad_blocks, g);
      note_launches(2);
    }
    return e;
  };
  if (g.linear) return act.dt == 0 ? launch(dw_split_kernel<0, 0>) : launch(dw_split_kernel<1, 0>);
  if (g.stride == 1) return act.dt == 0 ? launch(dw_split_kernel<0, 1>) : launch(dw_split_kernel<1, 1>);
  return act.dt == 0 ? launch(dw_split_kernel<0, 2>) : launch(dw_split_kernel<1, 2>);
}

}  // namespace surgeon
