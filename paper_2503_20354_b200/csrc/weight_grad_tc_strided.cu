// Tensor-core weight gradient of convolutions whose im2col operand has to be expanded: stride 2 and
// more, and the small-channel layers the direct kernel leaves (weight_grad_tc_direct.cu).
// Algorithm 1: Reshape and gradient steps with Eq. 2; the GEMM view of weight_grad_tc.cu:
//   D[nn, o] = sum_k Acol[nn, k] * G[o, k],  nn = (c, r, s),  k = (b, y, x), output rows padded to OWp,
// a multiple of 8 positions, so that a chunk of 8 positions (16 bytes of the operand) lies in one row.
//
// The output gradient is converted to bf16 by a pre-pass (padded rows, zeros in the padding) and
// arrives by TMA.  The activation operand is built by two groups of 8 warps in turns, a macro of a few
// K-tiles at a time:
//   1. the input rows that the macro's positions touch are rebuilt from the store in a shared-memory
//      patch, one lane per 16 elements of a row, once for all taps.  A row is kept as `stride` phase
//      planes (column ix goes to plane ix mod stride, place ix div stride), with zeros around:
//      what a tap reads for consecutive output positions is then consecutive, whatever the stride.  For strides 1 and 2
//      a lane's elements are whole 16-byte vectors of the planes, put together in registers;
//   2. a thread copies one chunk of 8 positions of four operand rows per K-tile: the 16 bytes that the chunk begins in and,
//      for a tap off a whole vector's start, the next 16, put in place by selects and a funnel shift.  Rows of the patch have
//      a pitch that spreads the eight lanes of such a load over the banks (five 4-byte loads, 16 bytes from lane to lane and
//      rows on the same banks, took 1440-2640 clocks a K-tile for what now takes 1040-1180).
// One group rebuilds while the other copies; the words and the values of a macro's first pieces are
// fetched while the macro before it is copied.  Bound by the instructions of the two steps, 430 for a warp's 32 pieces and
// 200 for its part of a K-tile: with 16 warps an SM issues at 0.53-0.57 of its rate and each warp every 8 clocks, for no one
// reason above a quarter; tensor pipe 11-15 %, DRAM 6-16 % busy (3x3 on 56x56 and the 7x7 stem, 70 % pruned).  So divisions are multiplications (also the
// sixteen of a thread's start: with them and branches in the fetch of a piece's words, a call of 15-21 us took 2 more), the
// copy and the fetch have no branches, a kept value costs one test for its load and its count, and a piece is put together in registers, not scattered bit by bit.
// Calls, 70 % pruned, when bits were scattered, with 4-byte copies, and now: 128 -> 128 channels on 56x56, batch 64, bf16
// 132, 94, 87 us; 256 -> 256 on 28x28 91, 73, 58; 512 -> 512 on 14x14 85, 68, 57; 160 -> 320 on 32x32, batch 200, fp32 179,
// 148, 113; 320 -> 640 on 16x16 171, 126, 105; 7x7 stride 2 on 224x224, 3 -> 64, batch 64, bf16 192, 161, 141 (two
// row tiles in a CTA).
// Every wait is bounded and ends in SURGEON_ERR_TIMEOUT.
#include <cuda.h>

#include <algorithm>

#include "surgeon_internal.cuh"
#include "tc_common.cuh"
#include "weight_grad_tc_conv.cuh"

namespace surgeon {

namespace {

using namespace tc;

constexpr int kTileM = 128;
constexpr int kTileK = 64;
constexpr int kGroups = 2;
constexpr int kGroupWarps = 8;
constexpr int kGroupThreads = kGroupWarps * 32;
constexpr int kThreads = 64 + kGroups * kGroupThreads;    // warp 0: MMA, warp 1: TMA, then the groups
constexpr int kMaxStages = 8;
constexpr int kATileBytes = kTileM * kTileK * 2;
constexpr int kMaxPatchBytes = 46 * 1024;                 // per group
constexpr int kPiece = 16;                                // elements of a row that one lane rebuilds

__device__ __forceinline__ void group_sync(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(kGroupThreads) : "memory");
}

// 16 bytes of shared memory: read, read where wanted (else zeros), written
__device__ __forceinline__ uint4 ld_shared_vec(uint32_t addr) {
  uint4 r;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(addr));
  return r;
}
__device__ __forceinline__ uint4 ld_shared_vec_if(uint32_t addr, bool wanted) {
  uint4 r;
  asm volatile("{.reg .pred q; setp.ne.u32 q, %5, 0; mov.u32 %0, 0; mov.u32 %1, 0; mov.u32 %2, 0; mov.u32 %3, 0;"
               "@q ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];}"
               : "=&r"(r.x), "=&r"(r.y), "=&r"(r.z), "=&r"(r.w) : "r"(addr), "r"(static_cast<uint32_t>(wanted)));
  return r;
}
__device__ __forceinline__ void st_shared_vec(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// The next packed value where the element's bit is set, else zero: one test for the load and the count
template <int DT>
__device__ __forceinline__ uint32_t take_next(const void* __restrict__ values, uint32_t& rank, uint32_t bit) {
  uint32_t r;
  const unsigned char* src = static_cast<const unsigned char*>(values) + static_cast<size_t>(rank) * (DT == 0 ? 4 : 2);
  if (DT == 0)
    asm volatile("{.reg .pred q; setp.ne.u32 q, %3, 0; mov.u32 %0, 0; @q ld.global.nc.u32 %0, [%2]; @q add.u32 %1, %1, 1;}"
                 : "=&r"(r), "+r"(rank) : "l"(src), "r"(bit));
  else
    asm volatile("{.reg .pred q; setp.ne.u32 q, %3, 0; mov.u32 %0, 0; @q ld.global.nc.u16 %0, [%2]; @q add.u32 %1, %1, 1;}"
                 : "=&r"(r), "+r"(rank) : "l"(src), "r"(bit));
  return r;
}

// A piece whose values are on their way: one predicated load per element (consecutive lanes have consecutive pieces of
// a channel, whose packed values lie in few cache lines).
struct PieceValues {
  uint32_t v[kPiece];
  uint32_t dst, col, len;                                 // place
  int m;                                                  // macro
};
template <int DT>
__device__ __forceinline__ uint32_t pair(uint32_t lo, uint32_t hi) {
  return DT == 0 ? pack_bf16x2(__uint_as_float(lo), __uint_as_float(hi)) : lo | (hi << 16);
}
// Into the row's phase planes.  The places of a piece are whole 16-byte vectors for strides 1 and 2; past the row's
// end they are zeros like the elements there.
template <int DT>
__device__ __forceinline__ void place(const PieceValues& q, uint32_t row, int stride, int plane, uint32_t inv_stride) {
  const uint32_t (&v)[kPiece] = q.v;
  if (stride == 1) {
    const uint32_t to = row + 2 * q.col;
    st_shared_vec(to, make_uint4(pair<DT>(v[0], v[1]), pair<DT>(v[2], v[3]), pair<DT>(v[4], v[5]), pair<DT>(v[6], v[7])));
    st_shared_vec(to + 16, make_uint4(pair<DT>(v[8], v[9]), pair<DT>(v[10], v[11]), pair<DT>(v[12], v[13]), pair<DT>(v[14], v[15])));
  } else if (stride == 2) {
#pragma unroll
    for (int ph = 0; ph < 2; ++ph)
      st_shared_vec(row + 2 * ph * plane + q.col,
                    make_uint4(pair<DT>(v[ph], v[ph + 2]), pair<DT>(v[ph + 4], v[ph + 6]), pair<DT>(v[ph + 8], v[ph + 10]),
                               pair<DT>(v[ph + 12], v[ph + 14])));
  } else {
    uint32_t at = (q.col * inv_stride) >> 16, ph = q.col - at * stride;           // col / stride
#pragma unroll
    for (int e = 0; e < kPiece; ++e) {
      if (static_cast<uint32_t>(e) < q.len)
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(row + 2 * (ph * plane + at)), "h"(static_cast<unsigned short>(pair<DT>(v[e], 0u))) : "memory");
      if (++ph == static_cast<uint32_t>(stride)) { ph = 0; ++at; }
    }
  }
}

// What a lane fetches for its piece: the kept count before the 128-element block the piece starts in, the
// block's words and the one after the piece's; and where the piece goes.
struct PieceRaw {
  uint32_t off, next, start, len;
  uint4 words;
  uint32_t dst, col;       // patch element of the row's first column, the piece's first column
  int m;                   // its macro
};

// MA: row tiles of a CTA, each an accumulator of 128 rows
template <int DT, int MA>
__global__ void __launch_bounds__(kThreads, 1)
dw_strided_kernel(const uint32_t* __restrict__ bitmap, const void* __restrict__ values,
                  const uint32_t* __restrict__ offsets, const __grid_constant__ CUtensorMap grad_map,
                  float* __restrict__ partial, uint32_t* __restrict__ status, StridedParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int n_cols = p.acc_n * p.n_acc;
  const int a_bytes = MA == 1 ? kATileBytes : p.a_bytes, stage_bytes = a_bytes + n_cols * 128;
  __shared__ __align__(8) unsigned long long bars[2 * kMaxStages + 1];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile uint32_t fail;

  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const uint32_t lane = lane_id();
  const int nn0 = blockIdx.x * p.rows_per_tile;           // the im2col rows are spread evenly over the row tiles
  const int nn_end = min(nn0 + p.rows_per_tile, p.n_gemm);
  const int o0 = blockIdx.y * n_cols;
  const int n_acc_here = min(p.n_acc, (p.O - o0 + p.acc_n - 1) / p.acc_n);
  const int split = blockIdx.z;
  const int m_begin = split * p.macros_per_split;
  const int m_end = min(m_begin + p.macros_per_split, p.total_macros);
  // K-tiles of macro m (the last one of an image may be short)
  auto tiles_of = [&](int m) {
    const int k = m - static_cast<int>(divide(m, p.by_macros)) * p.macros_per_img;
    return min(p.macro, p.tiles_per_img - k * p.macro);
  };

  const uint32_t full_bar = smem_u32(bars);
  const uint32_t empty_bar = smem_u32(bars + kMaxStages);
  const uint32_t acc_bar = smem_u32(bars + 2 * kMaxStages);
  if (tid == 0) {
    tma_prefetch_desc(&grad_map);
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(full_bar + 8 * s, kGroupWarps + 1);       // a group's warps + the TMA thread
      mbar_init(empty_bar + 8 * s, 1);
    }
    mbar_init(acc_bar, 1);
    fail = 0;
    fence_barrier_init();
  }
  if (warp == 0) tmem_alloc(smem_u32(&tmem_slot), p.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  pdl_trigger();                         // the split reduction may be launched; it waits for this grid

  if (warp == 0) {
    // ================= MMA issuer =================
    if (lane == 0) {
      const uint32_t idesc = make_idesc(kTileM, p.acc_n);
      const uint32_t smem0 = smem_u32(smem);
      const uint64_t a_base = make_desc(smem0), b_base = make_desc(smem0 + a_bytes);
      const uint64_t stage_inc = static_cast<uint64_t>(stage_bytes >> 4);
      const uint64_t acc_inc = static_cast<uint64_t>((p.acc_n * 128) >> 4);
      uint64_t da = a_base, db = b_base;
      uint32_t parity = 0, accum = 0;
      int s = 0;
      bool ok = true;
      for (int m = m_begin; m < m_end && ok; ++m) {
        for (int t = tiles_of(m); t > 0; --t) {
          ok = mbar_wait_suspend(full_bar + 8 * s, parity);
          if (!ok) break;
          tc_fence_after();
          if (MA == 2) {
            umma_ktile<1, 2>(tmem_base, p.acc_n, da, db, acc_inc, idesc, accum);
            umma_ktile<1, 2>(tmem_base + n_cols, p.acc_n, da + (kATileBytes >> 4), db, acc_inc, idesc, accum);
          } else if (n_acc_here == 1) umma_ktile<1, 2>(tmem_base, p.acc_n, da, db, acc_inc, idesc, accum);
          else umma_ktile<2, 2>(tmem_base, p.acc_n, da, db, acc_inc, idesc, accum);
          umma_commit(empty_bar + 8 * s);
          accum = 1;
          if (++s == p.stages) { s = 0; parity ^= 1; da = a_base; db = b_base; }
          else { da += stage_inc; db += stage_inc; }
        }
      }
      if (!ok) { fail = 1; atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT)); }
      umma_commit(acc_bar);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ================= gradient tiles by TMA =================
    if (lane == 0) {
      pdl_wait();                                  // the bf16 gradient copy is complete
      int s = 0;
      uint32_t round = 0;
      bool ok = true;
      for (int m = m_begin; m < m_end && ok; ++m) {
        const int img = divide(m, p.by_macros);
        const int kt0 = (m - img * p.macros_per_img) * p.macro;
        const int n_t = tiles_of(m);
        for (int t = 0; t < n_t; ++t) {
          if (round > 0 && !mbar_wait_suspend(empty_bar + 8 * s, (round - 1) & 1)) {
            fail = 1;
            atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
            ok = false;
            break;
          }
          const uint32_t b_addr = smem_u32(smem + s * stage_bytes + a_bytes);
          mbar_arrive_expect_tx(full_bar + 8 * s, static_cast<uint32_t>(n_acc_here * p.acc_n) * 128u);
          for (int a = 0; a < n_acc_here; ++a)
            tma_load_3d(b_addr + a * p.acc_n * 128, &grad_map, (kt0 + t) * kTileK, o0 + a * p.acc_n, img,
                        full_bar + 8 * s);
          if (++s == p.stages) { s = 0; ++round; }
        }
      }
    }
    __syncwarp();
  } else {
    // ================= producers =================
    const int g = (warp - 2) / kGroupWarps;
    const int gtid = tid - 64 - g * kGroupThreads;
    unsigned char* patch = smem + p.stages * stage_bytes + g * p.patch_bytes;
    const uint32_t smem_addr = smem_u32(smem), patch_addr = smem_u32(patch);
    const int c_first = nn0 / p.RS;
    const int c_last = (nn_end - 1) / p.RS;
    const int n_ch = c_last - c_first + 1;
    const int row_len = p.row_len;                 // elements of one input row in the patch, a multiple of 8
    // this thread's operand rows, 32 apart, and its chunk of 8 positions
    const int chunk = gtid & 7;
    // of row i: the 16 bytes of the patch that its column 0 of output row 0 begins in (with row_r input rows above the
    // patch's first), how many elements in, and the kernel row, -1000000 past the last column
    constexpr int kRows = 4 * MA;
    uint32_t row_addr[kRows], row_off[kRows];
    int row_r[kRows];
    const uint32_t dst_off = tile_off(gtid >> 3, chunk);   // (32 rows are 4 KB)
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int nn = nn0 + (gtid >> 3) + 32 * i;
      row_addr[i] = patch_addr;
      row_off[i] = 0;
      row_r[i] = -1000000;
      if (nn < nn_end) {
        const int c = divide(nn, p.by_rs), rs = nn - c * p.RS;
        const int r = divide(rs, p.by_kw), s = rs - r * p.KW;
        const int d = s - p.pad;
        const int fd = static_cast<int>(divide(d + 8 * p.stride, p.by_stride)) - 8;     // rounded down; pad <= 8 stride
        const int base = (c - c_first) * p.patch_rows * row_len + (d - fd * p.stride) * p.plane + 8 + fd;
        row_r[i] = r - p.pad;
        row_off[i] = base & 7;
        row_addr[i] = patch_addr + 2 * ((base & ~7) + row_r[i] * row_len);
      }
    }
    // Rows past the tile's share stay zero in every stage; the second of two tiles ends with its share, and what the
    // MMA reads past it goes to accumulator rows that nothing reads.
    const int n_mine = max(0, min(kRows, (p.rows_per_tile - (gtid >> 3) + 31) / 32));
    if (MA == 1)
      for (int st = 0; st < p.stages; ++st)
        for (int i = n_mine; i < kRows; ++i) st_shared_vec(smem_addr + st * stage_bytes + dst_off + i * 4096, make_uint4(0, 0, 0, 0));
    // A macro's pieces (channel, row, 16 columns), as many as its patch has; some rows may lie past the map.
    const uint32_t per_row = (p.W + kPiece - 1) / kPiece, per_ch = p.patch_rows * per_row, n_pieces = n_ch * per_ch;
    struct Macro { int kt0, n_t, iy_lo; uint32_t start; };
    auto geometry = [&](int m) {
      Macro q;
      const int img = divide(m, p.by_macros);
      q.kt0 = (m - img * p.macros_per_img) * p.macro;
      q.n_t = min(p.macro, p.tiles_per_img - q.kt0);
      q.iy_lo = max(static_cast<int>(divide(q.kt0 * kTileK, p.by_owp)) * p.stride - p.pad, 0);
      q.start = (static_cast<uint32_t>(img) * p.C + c_first) * (p.H * p.W) + q.iy_lo * p.W;
      return q;
    };
    auto fetch = [&](const Macro& q, uint32_t t) {
      PieceRaw r;
      const uint32_t ci = divide(t, p.by_ch), rest = t - ci * per_ch, row = divide(rest, p.by_row);
      r.col = (rest - row * per_row) * kPiece;
      r.dst = (ci * p.patch_rows + row) * row_len + 8;
      const bool live = t < n_pieces && q.iy_lo + static_cast<int>(row) < p.H;   // (else nothing kept, at element 0)
      r.start = live ? q.start + ci * (p.H * p.W) + row * p.W + r.col : 0u;
      r.len = live ? min(static_cast<uint32_t>(kPiece), p.W - r.col) : 0u;
      const uint32_t blk = r.start >> kBlockShift, wi = r.start >> 5;
      r.off = __ldg(offsets + blk);
      if (blk != p.partial_blk) {
        r.words = __ldg(reinterpret_cast<const uint4*>(bitmap) + blk);
      } else {                                     // the last, partial block of the bitmap
        const uint32_t w0 = blk * kBlockWords;
        r.words.x = __ldg(bitmap + w0);
        r.words.y = (w0 + 1 < p.n_words) ? __ldg(bitmap + w0 + 1) : 0u;
        r.words.z = (w0 + 2 < p.n_words) ? __ldg(bitmap + w0 + 2) : 0u;
        r.words.w = (w0 + 3 < p.n_words) ? __ldg(bitmap + w0 + 3) : 0u;
      }
      // (within the block the next word is at hand)
      r.next = ld_packed<0>(bitmap, wi + 1, (wi & 3u) == 3u && (r.start & 31u) + r.len > 32u);
      r.m = 0x7FFFFFFF;
      return r;
    };
    int s = 0;
    uint32_t round = 0;
    auto skip_tiles = [&](int n) {                 // the other group's
      s += n;
      while (s >= p.stages) { s -= p.stages; ++round; }
    };
    if (g == 1 && m_begin < m_end) skip_tiles(tiles_of(m_begin));
    auto wait_stage = [&]() {
      // (once a wait has given up nothing waits any more: the warps still meet at the group's barriers,
      // and what they write is not used)
      if (round > 0 && lane == 0 && !fail && !mbar_wait_suspend(empty_bar + 8 * s, (round - 1) & 1)) {
        fail = 1;
        atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
      }
    };
    // The thread's pieces are one stream over the group's macros: the words of a piece are fetched while the
    // values of the one before it are on their way, and those while the one before that is placed.
    // What is fetched ahead at a macro's end hides behind the copying of its operand tiles.
    int fm = m_begin + g;                          // macro and index of the next piece to fetch
    uint32_t ft = gtid;
    Macro fq = geometry(fm < m_end ? fm : m_begin);
    auto fetch_next = [&]() {
      if (ft >= n_pieces && fm < m_end) {         // (a thread past all pieces of a macro has none in the others either)
        fm = gtid < n_pieces ? fm + kGroups : m_end;
        ft = gtid;
        if (fm < m_end) fq = geometry(fm);
      }
      PieceRaw r = fetch(fq, fm < m_end ? ft : 0xFFFFFFFFu);
      if (fm < m_end) { r.m = fm; ft += kGroupThreads; }
      return r;
    };
    auto issue = [&](const PieceRaw& r, PieceValues& v) {
      const uint32_t wq = (r.start >> 5) & 3u, sh = r.start & 31u;
      uint32_t rank = r.off;
      rank += wq > 0 ? __popc(r.words.x) : 0u;
      rank += wq > 1 ? __popc(r.words.y) : 0u;
      rank += wq > 2 ? __popc(r.words.z) : 0u;
      const uint32_t w0 = wq == 0 ? r.words.x : (wq == 1 ? r.words.y : (wq == 2 ? r.words.z : r.words.w));
      const uint32_t w1 = wq == 3 ? r.next : (wq == 0 ? r.words.y : (wq == 1 ? r.words.z : r.words.w));
      rank += __popc(w0 & ((1u << sh) - 1u));
      const uint32_t bits = __funnelshift_r(w0, w1, sh) & ((1u << r.len) - 1u);
      // A fully kept piece (all of an unpruned tensor, the head of one whose zeros are kept in part) is consecutive values,
      // four at a time where they begin at a multiple of four.  (Eight bf16 values at a time leave the last piece of a row of 28
      // out, and its warp does both: 54 -> 58 us for 256 channels, batch 64.)
      if (bits == (1u << r.len) - 1u && (r.len == 0 || ((rank | r.len) & 3u) == 0)) {
        const unsigned char* src = static_cast<const unsigned char*>(values) + static_cast<size_t>(rank) * (DT == 0 ? 4 : 2);
#pragma unroll
        for (uint32_t j = 0; j < kPiece / 4; ++j) {
          const bool some = 4 * j < r.len;
          if (DT == 0) {
            const uint4 q = some ? __ldg(reinterpret_cast<const uint4*>(src) + j) : make_uint4(0, 0, 0, 0);
            v.v[4 * j] = q.x; v.v[4 * j + 1] = q.y; v.v[4 * j + 2] = q.z; v.v[4 * j + 3] = q.w;
          } else {
            const uint2 q = some ? __ldg(reinterpret_cast<const uint2*>(src) + j) : make_uint2(0, 0);
            v.v[4 * j] = q.x & 0xFFFFu; v.v[4 * j + 1] = q.x >> 16; v.v[4 * j + 2] = q.y & 0xFFFFu; v.v[4 * j + 3] = q.y >> 16;
          }
        }
      } else {
#pragma unroll
        for (int e = 0; e < kPiece; ++e) v.v[e] = take_next<DT>(values, rank, bits & (1u << e));
      }
      v.dst = r.dst; v.col = r.col; v.len = r.len; v.m = r.m;
    };
    PieceValues ready;
    PieceRaw raw = fetch_next();
    issue(raw, ready);
    raw = fetch_next();
    // (what no piece writes stays zero: the places around the rows)
    for (int v = gtid; v < p.patch_bytes / 16; v += kGroupThreads)
      reinterpret_cast<uint4*>(patch)[v] = make_uint4(0, 0, 0, 0);
    group_sync(g);
    for (int m = m_begin + g; m < m_end; m += kGroups) {
      const Macro q = geometry(m);
      const int kt0 = q.kt0, n_t = q.n_t, iy_lo = q.iy_lo;
      // ---- the patch ----
      while (ready.m == m) {
        place<DT>(ready, patch_addr + 2 * ready.dst, p.stride, p.plane, p.inv_stride);
        issue(raw, ready);
        raw = fetch_next();
      }
      group_sync(g);
      // ---- the operand tiles ----
      for (int t = 0; t < n_t; ++t) {
        wait_stage();
        __syncwarp();
        const uint32_t a_tile = smem_addr + s * stage_bytes;
        const int pos = (kt0 + t) * kTileK + 8 * chunk;
        const int y = divide(pos, p.by_owp), x0 = pos - y * p.OWp;
        const int nv = pos < p.P ? p.OW - x0 : 0;          // positions of the chunk that exist
        uint32_t keep[4];                                  // (the padding at the end of the row is zero)
#pragma unroll
        for (int j = 0; j < 4; ++j) keep[j] = nv > 2 * j + 1 ? 0xFFFFFFFFu : (nv == 2 * j + 1 ? 0xFFFFu : 0u);
        const int y_in = nv > 0 ? y * p.stride : -1000000;
        const uint32_t from = 2 * (x0 + (y_in - iy_lo) * row_len);
        // (all loads of two rows before the first store; rows at a whole vector's start need no second one; the patch
        // begins with zeros, which stand for what lies outside)
#pragma unroll
        for (int h = 0; h < kRows; h += 2) {
          if (h >= n_mine) break;
          uint4 lo[2], hi[2];
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            const bool in = static_cast<uint32_t>(y_in + row_r[h + k]) < static_cast<uint32_t>(p.H);
            const uint32_t addr = in ? row_addr[h + k] + from : patch_addr;
            lo[k] = ld_shared_vec(addr);
            hi[k] = ld_shared_vec_if(addr + 16, in && row_off[h + k] != 0);
          }
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (h + k >= n_mine) break;
            const uint32_t off = row_off[h + k];
            const uint32_t w[8] = {lo[k].x, lo[k].y, lo[k].z, lo[k].w, hi[k].x, hi[k].y, hi[k].z, hi[k].w};
            uint32_t q4[6], q2[5];
#pragma unroll
            for (int j = 0; j < 6; ++j) q4[j] = off & 4 ? w[j + 2] : w[j];
#pragma unroll
            for (int j = 0; j < 5; ++j) q2[j] = off & 2 ? q4[j + 1] : q4[j];
            const uint32_t shift = (off & 1) * 16;
            st_shared_vec(a_tile + dst_off + (h + k) * 4096,
                          make_uint4(__funnelshift_r(q2[0], q2[1], shift) & keep[0], __funnelshift_r(q2[1], q2[2], shift) & keep[1],
                                     __funnelshift_r(q2[2], q2[3], shift) & keep[2], __funnelshift_r(q2[3], q2[4], shift) & keep[3]));
          }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) mbar_arrive(full_bar + 8 * s);
        skip_tiles(1);
      }
      if (m + 1 < m_end) skip_tiles(tiles_of(m + 1));
      group_sync(g);                               // the patch is read; the next one takes its place
    }
  }

  // ================= epilogue: TMEM -> scratch partial tile =================
  if (warp >= 2) {
    const bool done = mbar_wait(acc_bar, 0, 64);
    tc_fence_after();
    if (done && !fail) {
      const int lane_grp = warp & 3;              // TMEM lanes this warp may read
      float* out = partial + static_cast<long long>(split) * p.O * p.n_gemm;
      const int cols_here = n_acc_here * p.acc_n;
#pragma unroll
      for (int m = 0; m < MA; ++m) {
        const int nn = nn0 + m * kTileM + lane_grp * 32 + static_cast<int>(lane);
        if (MA == 2 && nn - static_cast<int>(lane) >= nn_end) break;
        for (int col = 16 * ((warp - 2) >> 2); col < cols_here; col += 16 * (kGroups * kGroupWarps / 4)) {
          uint32_t r[16];
          tmem_ld16(tmem_base + (static_cast<uint32_t>(lane_grp * 32) << 16) + m * n_cols + col, r);
          if (nn < nn_end) {
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const int o = o0 + col + e;
              if (o < p.O && SURGEON_IN_BOUNDS(static_cast<long long>(split) * p.O * p.n_gemm +
                                                   static_cast<long long>(o) * p.n_gemm + nn,
                                               static_cast<long long>(p.splits) * p.O * p.n_gemm, status))
                out[static_cast<long long>(o) * p.n_gemm + nn] = __uint_as_float(r[e]);
            }
          }
        }
      }
    } else if (!done && lane == 0) {
      atomicMax(status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem_base, p.tmem_cols);
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                              CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                              CUtensorMapFloatOOBfill);

bool compute_plan_strided(const surgeon_layer_desc& d, StridedParams* out) {
  if (d.kind != 1) return false;
  StridedParams p{};
  p.B = d.batch; p.C = d.c_in; p.H = d.h; p.W = d.w; p.O = d.c_out; p.KH = d.kh; p.KW = d.kw;
  p.stride = d.stride; p.pad = d.pad;
  p.OH = (d.h + 2 * d.pad - d.kh) / d.stride + 1;
  p.OW = (d.w + 2 * d.pad - d.kw) / d.stride + 1;
  p.OWp = (p.OW + 7) / 8 * 8;
  p.P = p.OH * p.OWp;
  p.RS = d.kh * d.kw;
  p.n_gemm = d.c_in * p.RS;
  // 8 zeros to the left of a plane: tap columns reach at most 8 places over the edge; ix / stride by a multiplication
  if ((d.pad + d.stride - 1) / d.stride > 8 || (d.kw - 1) / d.stride > 5 || d.stride > 64 || d.w > 4096) return false;
  p.inv_stride = (65536 + d.stride - 1) / d.stride;
  for (int ix = 0; ix < d.w; ++ix)
    if (static_cast<int>((static_cast<unsigned>(ix) * p.inv_stride) >> 16) != ix / d.stride) return false;
  // elements of a plane: 8 zeros, then the row's pieces or what its last chunk reads, whichever is longer, in whole
  // 16-byte vectors
  const int pieces = (d.w + kPiece - 1) / kPiece * kPiece;
  p.plane = (std::max(p.OWp + 16, 8 + (pieces - 1) / d.stride + 1) + 7) / 8 * 8;
  // Pitch of the patch's rows: eight lanes read the eight chunks of a K-tile at once, 16 bytes each, from one output row
  // or several; of the four next multiples of 8 elements the one that leaves the fewest of them on the same banks.
  // Where rows without padding allow a longer macro they have none.
  int least = 1 << 30, pitch = 0;
  for (int more = 0; more < 32; more += 8) {
    const int len = d.stride * p.plane + more;
    int clashes = 0, used[8] = {0};
    for (int k = 0; k < 8; ++k) {
      const int at = (8 * k / p.OWp) * d.stride * len + 8 * k % p.OWp;
      clashes += used[at / 8 % 8]++;
    }
    if (clashes < least) { least = clashes; pitch = len; }
  }
  p.tiles_per_img = (p.P + kTileK - 1) / kTileK;
  // columns: one or two accumulators of at most 256 columns, the fewest padded columns first
  int best_waste = -1;
  for (int c = 256; c >= 16; c -= 16) {
    const int units = (p.O + c - 1) / c;
    const int waste = units * c - p.O;
    if (best_waste < 0 || waste < best_waste) { best_waste = waste; p.acc_n = c; }
  }
  const int units = (p.O + p.acc_n - 1) / p.acc_n;
  // the longest macro (rows are rebuilt once per macro) whose patch fits, with three stages at least if possible
  const int budget = 226 * 1024 - 1024 - 256;
  bool found = false;
  // Between 129 and 256 rows one CTA takes them all, as two row tiles: one rebuild, one gradient tile, one round of
  // waits for both, instead of two CTAs with halves that need the channels between them twice.  Its start and its
  // epilogue are longer and there are twice the partial results, so only from 32 K-tiles an SM on: 3 -> 64 channels 7x7
  // stride 2 on 224x224, batch 64 (85 an SM), 161 -> 142 us; 16 -> 64 3x3 on 56x56, batch 64 (21), 54 -> 52; 16 -> 160 3x3 on
  // 32x32, batch 200 (22), 72.7 -> 74.8; the first at batch 4 (5) 25.6 -> 29.6.  Nor with 256 columns, where the copy is a smaller part of
  // a K-tile: 16 -> 256 on 56x56, batch 110 (36), 148.5 -> 150.6; 3 -> 160 7x7 (64) 189 -> 175.
  const bool pairs = p.n_gemm > kTileM && p.n_gemm <= 2 * kTileM && units == 1 && p.acc_n <= 192 &&
                     static_cast<long long>(d.batch) * p.tiles_per_img >= 32LL * sm_count();
  for (int m_acc = pairs ? 2 : 1; m_acc >= 1 && !found; --m_acc) {
    p.m_acc = m_acc;
    p.m_tiles = (p.n_gemm + m_acc * kTileM - 1) / (m_acc * kTileM);
    p.rows_per_tile = ((p.n_gemm + p.m_tiles - 1) / p.m_tiles + 7) / 8 * 8;
    p.a_bytes = m_acc == 1 ? kATileBytes : p.rows_per_tile * kTileK * 2;
    // channels a tile's rows can touch
    const int n_ch = p.rows_per_tile < 2 ? 1 : (p.C < (p.rows_per_tile - 2) / p.RS + 2 ? p.C : (p.rows_per_tile - 2) / p.RS + 2);
    for (int want_stages = 3; want_stages >= 2 && !found; --want_stages) {
      for (int n_acc = units >= 2 ? 2 : 1; n_acc >= 1 && !found; --n_acc) {
        for (int macro = 8; macro >= 1 && !found; --macro) {
          if (macro > p.tiles_per_img) continue;
          // (where macros begin with a row, whole rows)
          int out_rows = macro * kTileK % p.OWp == 0 ? macro * kTileK / p.OWp : (macro * kTileK + p.OWp - 2) / p.OWp + 1;
          if (out_rows > p.OH) out_rows = p.OH;
          int rows = (out_rows - 1) * d.stride + d.kh;
          if (rows > d.h) rows = d.h;
          for (int len : {pitch, d.stride * p.plane}) {
            const long long bytes = (static_cast<long long>(n_ch) * rows * len * 2 + 32 + 15) / 16 * 16;
            if (bytes > kMaxPatchBytes) continue;
            const int stage = p.a_bytes + n_acc * p.acc_n * 128;
            int stages = static_cast<int>((budget - kGroups * bytes) / stage);
            if (stages > kMaxStages) stages = kMaxStages;
            if (stages < want_stages || macro >= stages) continue;    // (macro < stages: see the producers' waits)
            // (the MMAs read two whole row tiles of the last stage)
            if (m_acc == 2 && stage + kGroups * bytes < 2 * kATileBytes) continue;
            p.macro = macro; p.patch_rows = rows; p.row_len = len; p.patch_bytes = static_cast<int>(bytes);
            p.n_acc = n_acc; p.stages = stages;
            found = true;
            break;
          }
        }
      }
    }
  }
  if (!found) return false;
  p.n_tiles = (units + p.n_acc - 1) / p.n_acc;
  p.macros_per_img = (p.tiles_per_img + p.macro - 1) / p.macro;
  const int per_row = (d.w + kPiece - 1) / kPiece;
  p.by_row = make_div(per_row); p.by_ch = make_div(per_row * p.patch_rows);
  p.by_rs = make_div(p.RS); p.by_kw = make_div(d.kw); p.by_stride = make_div(d.stride);
  p.by_owp = make_div(p.OWp); p.by_macros = make_div(p.macros_per_img);
  const long long total = static_cast<long long>(d.batch) * p.macros_per_img;
  if (total > 2147483647LL / 64) return false;
  p.total_macros = static_cast<int>(total);
  const int sms = sm_count();
  const long long tiles_mn = static_cast<long long>(p.m_tiles) * p.n_tiles;
  int best = 1;
  double best_cost = 1e30;
  for (int s = 1; s <= p.total_macros && s <= 160; ++s) {
    const long long waves = (tiles_mn * s + sms - 1) / sms;
    const int per = (p.total_macros + s - 1) / s;
    const double cost = static_cast<double>(waves) * (per * p.macro + 10) + 0.02 * s * tiles_mn / sms;
    if (cost < best_cost - 1e-9) { best_cost = cost; best = s; }
  }
  p.macros_per_split = (p.total_macros + best - 1) / best;
  p.splits = (p.total_macros + p.macros_per_split - 1) / p.macros_per_split;
  p.tmem_cols = 32;
  while (p.tmem_cols < p.acc_n * p.n_acc * p.m_acc) p.tmem_cols *= 2;
  p.smem_bytes = p.stages * (p.a_bytes + p.n_acc * p.acc_n * 128) + kGroups * p.patch_bytes + 1024;
  *out = p;
  return true;
}

}  // namespace

bool plan_strided(const surgeon_layer_desc& d, StridedParams* out) {
  struct Tag {};
  return memo_plan<Tag>(d, 0, out, [&](StridedParams* p) { return compute_plan_strided(d, p); });
}

size_t strided_partial_bytes(const StridedParams& p) {
  const size_t b = static_cast<size_t>(p.splits) * p.O * p.n_gemm * sizeof(float);
  return (b + 255) & ~static_cast<size_t>(255);
}

size_t strided_grad_bf16_bytes(const StridedParams& p) {
  const size_t b = static_cast<size_t>(p.B) * p.O * p.P * 2;
  return (b + 255) & ~static_cast<size_t>(255);
}

cudaError_t launch_strided(const surgeon_compressed& act, const StridedParams& plan, const float* grad_out,
                           void* grad_bf16, float* partial, uint32_t* status, cudaStream_t stream) {
  StridedParams p = plan;
  p.n_words = (act.n + 31) / 32;
  p.partial_blk = (act.n % SURGEON_BLOCK) ? static_cast<unsigned>(act.n / SURGEON_BLOCK) : 0xFFFFFFFFu;
  cudaError_t e = p.OW == p.OWp
                      ? launch_grad_to_bf16(grad_out, static_cast<long long>(p.B) * p.O * p.P, grad_bf16, status, stream)
                      : launch_grad_to_bf16_rows(grad_out, static_cast<long long>(p.B) * p.O * p.OH, p.OW, p.OWp,
                                                 grad_bf16, status, stream);
  if (e != cudaSuccess) return e;
  const EncodeFn encode = reinterpret_cast<EncodeFn>(tensor_map_encode_fn());
  if (!encode) return cudaErrorNotSupported;
  CUtensorMap map;
  const cuuint64_t dims[3] = {static_cast<cuuint64_t>(p.P), static_cast<cuuint64_t>(p.O),
                              static_cast<cuuint64_t>(p.B)};
  const cuuint64_t strides[2] = {static_cast<cuuint64_t>(p.P) * 2, static_cast<cuuint64_t>(p.P) * p.O * 2};
  const cuuint32_t box[3] = {static_cast<cuuint32_t>(kTileK), static_cast<cuuint32_t>(p.acc_n), 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  if (encode(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, grad_bf16, dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const dim3 grid(p.m_tiles, p.n_tiles, p.splits);
  auto launch = [&](auto kernel) -> cudaError_t {
    const cudaError_t err = allow_dynamic_smem(reinterpret_cast<const void*>(kernel), p.smem_bytes);
    if (err != cudaSuccess) return err;
    return launch_kernel(kernel, grid, dim3(kThreads), static_cast<size_t>(p.smem_bytes), stream, true, act.bitmap,
                         static_cast<const void*>(act.values), act.block_offsets, map, partial, status, p);
  };
  if (p.m_acc == 2) e = act.dt == 0 ? launch(dw_strided_kernel<0, 2>) : launch(dw_strided_kernel<1, 2>);
  else e = act.dt == 0 ? launch(dw_strided_kernel<0, 1>) : launch(dw_strided_kernel<1, 1>);
  note_launches(1);
  return e;
}

}  // namespace surgeon
