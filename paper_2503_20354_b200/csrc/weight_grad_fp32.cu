// fp32 path of surgeon_weight_grad (Algorithm 1: Reshape and gradient steps, Eq. 2): its launcher, and the kernel on CUDA
// cores, for the layers that the tensor cores (weight_grad_fp32_split.cu) do not take and the operands that they cannot hold.
//
// Implicit GEMM  dW[m, nn] = sum_k G[k, m] * Acol[k, nn]  with m = output channel,
// nn = (c, r, s) and k = (b, y, x) (or the row t of a linear layer).  The im2col operand is
// rebuilt from the compressed store straight into shared memory; the dense activation never exists
// in global memory.  The reduction is cut into chunks of at most 2048 terms; every chunk is summed in
// fp32 in a fixed order, and the chunk sums are added in double in a fixed order by a second
// kernel, so the result is reproducible and stays within ~3e-6 relative error of exact arithmetic.
//
// A CTA of 128 threads owns 64 x 128 outputs (8 x 8 per thread, packed two to an instruction) and
// works in K-tiles of 32 positions of one or more images: every thread rebuilds the 32 positions of one
// column - one rank computation per row of the map, then a bit test and a predicated load per
// element, or a rank per element where rows are shorter than four - and four CTAs per SM hide the
// latency of that behind one another's products.
// Measured on 320 -> 320 channels, 3x3 on 16x16, batch 16 (7.5 GFLOP): 1084 us with a rank
// computation per element and 4 x 4 outputs per thread, 264 us now: 28.6 TFLOP/s, 38 % of what the
// FMA pipes could do, since rebuilding and products take turns.  Small maps (128 -> 128 channels on
// 1x1, 200 000 images: 0.42 ms) and linear layers (4096 rows, 320 -> 320: 70 us) by elements.
#include <algorithm>
#include <type_traits>

#include "fp32_path.cuh"

namespace surgeon {

namespace {

constexpr int TM = 64, TN = 128, TK = 32;
constexpr int kThreads = 128;
constexpr int kCtasPerSm = 4;
constexpr int kMaxTiles = 2048 / TK;    // K-tiles of one chunk at most
constexpr int kGPitch = TM + 4, kAPitch = TN + 4;

struct Geom {
  int kind, B, C, H, W, O, KH, KW, stride, pad, OH, OW;
  int P;                 // positions per image (linear: rows)
  int by_element;        // conv: stretches of a row too short to be worth a rank computation each
  int k_tiles, per_chunk, chunks;
  int tiles_per_img;     // 0: K-tiles run over the images
  int K;                 // what the GEMM sums over
  long long M, N;        // its other extents
  long long n_words;
};

// What the tensor cores (weight_grad_fp32_split.cu) left behind, where they ran first.
struct SplitResult {
  const uint32_t* most;     // largest magnitudes: n_grad words of the gradient, n_act of the activation
  int* n_parts;             // to be set: partial sums per output, and whether they carry the factor of both operands
  int n_grad, n_act, chunks;
  uint32_t* status;         // the store's status word, for checked builds (set in either case)
};

// Whether the tensor cores' partial sums stand, given the bf16 patterns of the largest scaled magnitudes.  Infinities, NaN and
// what the factor makes infinite have no parts; a chunk's 2048 products, each below 2^(ea + eb - 2 * 127 + 2), have to
// stay below 2^127.  There is no lower limit: the factor gives every number its three parts (kSplitShift).
__device__ __forceinline__ bool split_holds(uint32_t a, uint32_t b) {
  if (a >= 0x7F80u || b >= 0x7F80u) return false;
  return (a >> 7) + (b >> 7) <= 2 * 127 + 127 - 11 - 2;    // (exponents, 127 more than they are)
}

Geom make_geom(const surgeon_layer_desc& d) {
  Geom g;
  g.kind = d.kind; g.B = d.kind == 1 ? d.batch : 1; g.C = d.c_in; g.H = d.h; g.W = d.w; g.O = d.c_out;
  g.KH = d.kh; g.KW = d.kw; g.stride = d.stride; g.pad = d.pad;
  g.OH = (d.h + 2 * d.pad - d.kh) / d.stride + 1;
  g.OW = (d.w + 2 * d.pad - d.kw) / d.stride + 1;
  g.P = d.kind == 1 ? g.OH * g.OW : d.batch;
  g.by_element = g.OW < 4 || 63 / d.stride + 1 < 4;
  // A K-tile stays inside an image, whose last one is partly used, unless that would leave more than a fifth of K
  // unused (or K beyond what the grid takes): 49 positions 772 -> 730 us, one position 5.7 -> 0.42 ms; at 196
  // positions (12 % unused) tiles over images cost 95 -> 100 us.
  const long long padded = (static_cast<long long>(g.P) + TK - 1) / TK * TK;
  const bool inside = 4 * padded <= 5LL * g.P && g.B * padded <= 65535LL * kMaxTiles * TK;
  g.tiles_per_img = inside ? static_cast<int>(padded / TK) : 0;
  const long long k_all = inside ? g.B * padded : static_cast<long long>(g.B) * g.P;
  g.k_tiles = static_cast<int>((k_all + TK - 1) / TK);
  g.K = static_cast<int>(k_all);
  g.M = d.c_out;
  g.N = static_cast<long long>(d.c_in) * d.kh * d.kw;
  g.n_words = (static_cast<long long>(d.batch) * d.c_in * d.h * d.w + 31) / 32;
  // K-tiles per chunk: as many rounds of resident CTAs as it takes, each as short as possible; a
  // chunk costs about two K-tiles (start, epilogue and its part of the reduction) on top of its own
  const long long tiles = ((g.M + TM - 1) / TM) * ((g.N + TN - 1) / TN);
  const long long slots = static_cast<long long>(kCtasPerSm) * sm_count();
  double best = 1e300;
  g.per_chunk = kMaxTiles;
  for (int per = 1; per <= kMaxTiles; ++per) {
    const long long chunks = (g.k_tiles + per - 1) / per;
    if (chunks > 65535) continue;                // (blockIdx.z)
    const long long waves = (tiles * chunks + slots - 1) / slots;
    const double cost = static_cast<double>(waves) * (per + 2.0);
    if (cost <= best) { best = cost; g.per_chunk = per; }
  }
  g.chunks = (g.k_tiles + g.per_chunk - 1) / g.per_chunk;
  return g;
}

// The value of packed element `idx` where `on`, else 0; widened to fp32.
template <int DT>
__device__ __forceinline__ float packed_value(const void* __restrict__ values, uint32_t idx, bool on) {
  if (DT == 0) return on ? __ldg(reinterpret_cast<const float*>(values) + idx) : 0.0f;
  const uint32_t h = on ? static_cast<uint32_t>(__ldg(reinterpret_cast<const unsigned short*>(values) + idx)) : 0u;
  return __uint_as_float(h << 16);
}

// The elements at flat indices j[i] (negative: zero).  First the words of all, then the values of all.
template <int DT, int N>
__device__ __forceinline__ void element_values(const uint32_t* __restrict__ bitmap, const void* __restrict__ values,
                                               const uint32_t* __restrict__ offsets, uint32_t n_words,
                                               const int (&j)[N], float (&v)[N]) {
  static_assert(kBlockWords == 4, "a block's words are one vector");
  uint4 q[N];
  uint32_t idx[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t blk = static_cast<uint32_t>(j[i]) >> kBlockShift, w0 = blk * kBlockWords;
    q[i] = make_uint4(0, 0, 0, 0);
    idx[i] = 0;
    if (j[i] >= 0) {
      idx[i] = __ldg(offsets + blk);
      if (w0 + 4 <= n_words) {
        q[i] = __ldg(reinterpret_cast<const uint4*>(bitmap) + blk);
      } else {                                     // the last, partial block
        q[i].x = __ldg(bitmap + w0);
        q[i].y = w0 + 1 < n_words ? __ldg(bitmap + w0 + 1) : 0u;
        q[i].z = w0 + 2 < n_words ? __ldg(bitmap + w0 + 2) : 0u;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const uint32_t wq = (static_cast<uint32_t>(j[i]) >> 5) & 3u, bit = static_cast<uint32_t>(j[i]) & 31u;
    const uint32_t w = wq == 0 ? q[i].x : (wq == 1 ? q[i].y : (wq == 2 ? q[i].z : q[i].w));
    idx[i] += (wq > 0 ? __popc(q[i].x) : 0) + (wq > 1 ? __popc(q[i].y) : 0) + (wq > 2 ? __popc(q[i].z) : 0) +
              __popc(w & ((1u << bit) - 1u));
    v[i] = packed_value<DT>(values, idx[i], ((w >> bit) & 1u) != 0u);
  }
}

// 64 bitmap bits from flat index j on, and the number of kept elements before j.
__device__ __forceinline__ unsigned long long bit_window(const uint32_t* __restrict__ bitmap,
                                                         const uint32_t* __restrict__ offsets,
                                                         long long n_words, long long j, uint32_t* rank) {
  const long long wi = j >> 5, blk = j >> kBlockShift;
  const uint32_t sh = static_cast<uint32_t>(j & 31);
  uint32_t r = __ldg(offsets + blk);
  const int before = static_cast<int>(wi - blk * kBlockWords);    // words of the block before the one of j
  const uint32_t p0 = before > 0 ? __ldg(bitmap + wi - before) : 0u;
  const uint32_t p1 = before > 1 ? __ldg(bitmap + wi - before + 1) : 0u;
  const uint32_t p2 = before > 2 ? __ldg(bitmap + wi - before + 2) : 0u;
  const uint32_t w0 = __ldg(bitmap + wi);
  const uint32_t w1 = wi + 1 < n_words ? __ldg(bitmap + wi + 1) : 0u;
  const uint32_t w2 = wi + 2 < n_words ? __ldg(bitmap + wi + 2) : 0u;
  r += __popc(p0) + __popc(p1) + __popc(p2) + __popc(w0 & ((1u << sh) - 1u));
  *rank = r;
  return (static_cast<unsigned long long>(__funnelshift_r(w1, w2, sh)) << 32) | __funnelshift_r(w0, w1, sh);
}

__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long twice(float v) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(v));
  return r;
}

// KIND: 0 linear, 1 convolution by stretches of a row, 2 convolution by elements (Geom::by_element).
// SPAN: K-tiles run over the images (Geom::tiles_per_img is 0).
template <int DT, int KIND, bool SPAN>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
dw_fp32_kernel(const uint32_t* __restrict__ bitmap, const void* __restrict__ values,
               const uint32_t* __restrict__ offsets, const float* __restrict__ grad,
               float* __restrict__ partial, Geom g, SplitResult split) {
  if (split.most) {                              // the tensor cores' result stands unless their planes could not hold an operand
    pdl_wait();
    __shared__ uint32_t s_most[2];
    if (threadIdx.x < 2) s_most[threadIdx.x] = 0;
    __syncthreads();
    uint32_t m[2] = {0, 0};
    for (int i = threadIdx.x; i < split.n_grad + split.n_act; i += kThreads) {
      uint32_t& x = m[i < split.n_grad ? 0 : 1];
      x = max(x, split.most[i]);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      m[i] = __reduce_max_sync(0xFFFFFFFFu, m[i]);
      if (lane_id() == 0) atomicMax(&s_most[i], m[i]);
    }
    __syncthreads();
    const bool stands = split_holds(s_most[0], s_most[1]);
    if (threadIdx.x == 0 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0) {
      split.n_parts[0] = stands ? split.chunks : g.chunks;
      split.n_parts[1] = stands ? 1 : 0;
    }
    pdl_trigger();
    if (stands) return;
  }
  __shared__ __align__(16) float Gs[TK][kGPitch];
  __shared__ __align__(16) float As[TK][kAPitch];
  const int tid = threadIdx.x;
  const long long m0 = static_cast<long long>(blockIdx.y) * TM;
  const long long n0 = static_cast<long long>(blockIdx.x) * TN;
  const int kt_begin = blockIdx.z * g.per_chunk;
  const int kt_end = min(kt_begin + g.per_chunk, g.k_tiles);
  // this thread's column of the activation tile
  const long long col = n0 + tid;
  const bool col_ok = col < g.N;
  int c = 0, r = 0, s = 0;
  if (KIND != 0 && col_ok) {
    const int RS = g.KH * g.KW;
    c = static_cast<int>(col / RS);
    const int rs = static_cast<int>(col - static_cast<long long>(c) * RS);
    r = rs / g.KW;
    s = rs - r * g.KW;
  }

  unsigned long long acc[8][4];                    // 8 output channels x 4 pairs of columns
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0ull;
  const int ty = tid >> 4, tx = tid & 15;
  const bool vec4 = (g.P & 3) == 0;                // four positions from a multiple of 4 on: one image, 16 bytes

  for (int kt = kt_begin; kt < kt_end; ++kt) {
    // the tile's first position: its image and its place there
    int img = KIND == 0 ? 0 : (SPAN ? kt * TK / g.P : kt / g.tiles_per_img);
    const int p0 = SPAN ? kt * TK - img * g.P : (kt - img * g.tiles_per_img) * TK;
    const int n_pos = min(TK, SPAN ? g.K - kt * TK : g.P - p0);
    const int n_used = KIND == 1 ? TK : (n_pos + 7) & ~7;      // rows of the tiles that the products read
    // ---- the gradient tile, transposed ----
    if (KIND != 0) {                               // [b][m][position]
      const int mm = tid >> 1, half = tid & 1;
      const float* src = grad + (static_cast<long long>(img) * g.O + m0 + mm) * g.P + p0;
      const bool ok = m0 + mm < g.M;
#pragma unroll
      for (int i = 0; i < 4; ++i) {                // (the two threads of a row alternate: no bank conflicts)
        const int k = 8 * i + 4 * half;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (SPAN && ok && k < n_pos) {
          int p = (p0 + k) % g.P;
          const float* at = src - p0 + static_cast<long long>((p0 + k) / g.P) * g.O * g.P + p;
          if (vec4) {                              // (n_pos is a multiple of 4 as well)
            v = __ldg(reinterpret_cast<const float4*>(at));
          } else {
            float* f = reinterpret_cast<float*>(&v);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              if (k + e < n_pos) f[e] = __ldg(at);
              ++at;
              if (++p == g.P) { p = 0; at += (g.O - 1LL) * g.P; }
            }
          }
        }
        if (!SPAN && ok) {
          if (vec4 && k + 4 <= n_pos) {
            v = __ldg(reinterpret_cast<const float4*>(src + k));
          } else {
            v.x = k < n_pos ? __ldg(src + k) : 0.0f;
            v.y = k + 1 < n_pos ? __ldg(src + k + 1) : 0.0f;
            v.z = k + 2 < n_pos ? __ldg(src + k + 2) : 0.0f;
            v.w = k + 3 < n_pos ? __ldg(src + k + 3) : 0.0f;
          }
        }
        Gs[k][mm] = v.x; Gs[k + 1][mm] = v.y; Gs[k + 2][mm] = v.z; Gs[k + 3][mm] = v.w;
      }
    } else {                                       // [row][m]
      const int mm = tid & (TM - 1);
#pragma unroll
      for (int i = 0; i < TK / 2; ++i) {
        const int k = 2 * i + (tid >> 6);
        Gs[k][mm] = (k < n_pos && m0 + mm < g.M) ? __ldg(grad + static_cast<long long>(p0 + k) * g.O + m0 + mm) : 0.0f;
      }
    }
    // ---- this thread's column of the activation tile ----
    if (KIND == 1) {
      int y = p0 / g.OW, x = p0 - y * g.OW;
      for (int k = 0; k < n_used;) {
        // a piece: positions of one output row, at most 64 input elements wide
        int len = n_used - k;
        uint32_t rank = 0;
        unsigned long long win = 0;
        if (k < n_pos) {
          len = min(min(n_pos - k, g.OW - x), 63 / g.stride + 1);
          const int iy = y * g.stride + r - g.pad;
          int ix = x * g.stride + s - g.pad;
          int skip = 0;                            // leading positions left of the map
          if (ix < 0) { skip = (-ix + g.stride - 1) / g.stride; ix += skip * g.stride; }
          // positions inside the map; the window's bits past them are dropped
          const int inside = ix < g.W ? min(len - skip, (g.W - 1 - ix) / g.stride + 1) : 0;
          if (col_ok && iy >= 0 && iy < g.H && inside > 0) {
            win = bit_window(bitmap, offsets, g.n_words,
                             ((static_cast<long long>(img) * g.C + c) * g.H + iy) * g.W + ix, &rank);
            const int bits = (inside - 1) * g.stride + 1;
            if (bits < 64) win &= (1ull << bits) - 1ull;
            win <<= skip * g.stride;
          }
        }
        const unsigned long long step_mask = (1ull << g.stride) - 1ull;    // (stride at most 21: see by_element)
        for (int e0 = 0; e0 < len; e0 += 8) {
          float v[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            v[e] = packed_value<DT>(values, rank, (win & 1ull) != 0ull);
            rank += g.stride == 1 ? static_cast<uint32_t>(win & 1ull) : static_cast<uint32_t>(__popcll(win & step_mask));
            win >>= g.stride;
          }
#pragma unroll
          for (int e = 0; e < 8; ++e)
            if (e0 + e < len) As[k + e0 + e][tid] = v[e];
        }
        k += len;
        x += len;
        if (x >= g.OW) {
          x = 0;
          ++y;
          if (SPAN && y == g.OH) { y = 0; ++img; }
        }
      }
    } else {
      int y = 0, x = 0;
      if (KIND == 2) { y = p0 / g.OW; x = p0 - y * g.OW; }
      constexpr int kAtOnce = 8;
#pragma unroll 1
      for (int k = 0; k < n_used; k += kAtOnce) {
        int j[kAtOnce];
        float v[kAtOnce];
#pragma unroll
        for (int e = 0; e < kAtOnce; ++e) {
          j[e] = -1;
          if (KIND == 0) {
            if (k + e < n_pos && col_ok) j[e] = (p0 + k + e) * g.C + static_cast<int>(col);
          } else {
            const int iy = y * g.stride + r - g.pad, ix = x * g.stride + s - g.pad;
            if (k + e < n_pos && col_ok && iy >= 0 && iy < g.H && ix >= 0 && ix < g.W)
              j[e] = ((img * g.C + c) * g.H + iy) * g.W + ix;
            if (++x == g.OW) {
              x = 0;
              ++y;
              if (SPAN && y == g.OH) { y = 0; ++img; }
            }
          }
        }
        element_values<DT>(bitmap, values, offsets, static_cast<uint32_t>(g.n_words), j, v);
#pragma unroll
        for (int e = 0; e < kAtOnce; ++e) As[k + e][tid] = v[e];
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < n_used; ++kk) {          // (a multiple of 8)
      const ulonglong2 a0 = *reinterpret_cast<const ulonglong2*>(&As[kk][tx * 4]);
      const ulonglong2 a1 = *reinterpret_cast<const ulonglong2*>(&As[kk][TN / 2 + tx * 4]);
      const float4 g0 = *reinterpret_cast<const float4*>(&Gs[kk][ty * 8]);
      const float4 g1 = *reinterpret_cast<const float4*>(&Gs[kk][ty * 8 + 4]);
      const float gr[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const unsigned long long gg = twice(gr[a]);
        fma2(acc[a][0], gg, a0.x);
        fma2(acc[a][1], gg, a0.y);
        fma2(acc[a][2], gg, a1.x);
        fma2(acc[a][3], gg, a1.y);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const long long m = m0 + ty * 8 + a;
    if (m >= g.M) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const long long nn = n0 + (b >> 1) * (TN / 2) + tx * 4 + (b & 1) * 2;
      const float lo = __uint_as_float(static_cast<uint32_t>(acc[a][b]));
      const float hi = __uint_as_float(static_cast<uint32_t>(acc[a][b] >> 32));
      const long long at = (blockIdx.z * g.M + m) * g.N + nn;
      if (nn < g.N && SURGEON_IN_BOUNDS(at, g.chunks * g.M * g.N, split.status)) partial[at] = lo;
      if (nn + 1 < g.N && SURGEON_IN_BOUNDS(at + 1, g.chunks * g.M * g.N, split.status)) partial[at + 1] = hi;
    }
  }
}

// The partial sums, in double, in a fixed order.  n_parts: how many there are (null: `chunks`), and whether the factor of
// both operands is taken out again (exact in double: no number is rounded twice).  V outputs a thread, or
// (V = 1, blocks of 32 x 8) one by eight threads, which take every eighth partial sum.
template <int V, bool EIGHT>
__global__ void __launch_bounds__(256)
reduce_chunks_kernel(const float* __restrict__ partial, long long mn, int chunks, const int* n_parts,
                     float* __restrict__ dw, int accumulate, uint32_t* status) {
  static_assert(V == 1 || !EIGHT, "one output");
  pdl_wait();
  double factor = 1.0;
  if (n_parts) {
    chunks = n_parts[0];
    if (n_parts[1]) factor = 1.0 / static_cast<double>(1ull << (2 * kSplitShift));
  }
  const long long i = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) * V;
  using Vec = typename std::conditional<V == 4, float4, float>::type;
  double s[V];
#pragma unroll
  for (int e = 0; e < V; ++e) s[e] = 0.0;
  if (i < mn) {
#pragma unroll 8
    for (int z = EIGHT ? threadIdx.y : 0; z < chunks; z += EIGHT ? 8 : 1) {
      const Vec v = __ldg(reinterpret_cast<const Vec*>(partial + z * mn + i));
#pragma unroll
      for (int e = 0; e < V; ++e) s[e] += static_cast<double>(reinterpret_cast<const float*>(&v)[e]);
    }
  }
  if (EIGHT) {
    __shared__ double part[8][32];
    part[threadIdx.y][threadIdx.x] = s[0];
    __syncthreads();
    if (threadIdx.y != 0) return;
#pragma unroll
    for (int y = 1; y < 8; ++y) s[0] += part[y][threadIdx.x];
  }
  if (i >= mn || !SURGEON_IN_BOUNDS(i + V - 1, mn, status)) return;
  float out[V];
#pragma unroll
  for (int e = 0; e < V; ++e) {
    s[e] *= factor;
    out[e] = accumulate ? static_cast<float>(static_cast<double>(dw[i + e]) + s[e]) : static_cast<float>(s[e]);
  }
  *reinterpret_cast<Vec*>(dw + i) = *reinterpret_cast<const Vec*>(out);
}

}  // namespace

// Scratch of a layer for the tensor cores: the count of partial sums per output and the largest magnitudes, the gradient's
// planes, then the partial sums.
static size_t split_head_bytes(const SplitGeom& s) {
  return (16 + (static_cast<size_t>(s.slabs) * s.grad_blocks + s.ctas) * 4 + 255) & ~static_cast<size_t>(255);
}

size_t weight_grad_fp32_workspace(const surgeon_layer_desc& d) {
  const Geom g = make_geom(d);
  SplitGeom s;
  const bool split = plan_split(d, &s);
  const int chunks = std::max(std::max(g.chunks, 1), split ? s.chunks : 0);
  return (split ? split_head_bytes(s) + split_planes_bytes(s) : 0) + static_cast<size_t>(chunks) * g.M * g.N * sizeof(float);
}

cudaError_t launch_weight_grad_fp32(const surgeon_compressed& act, const surgeon_layer_desc& d,
                                    const float* grad_out, float* dw, int accumulate,
                                    void* workspace, cudaStream_t stream) {
  const Geom g = make_geom(d);
  float* partial = static_cast<float*>(workspace);
  SplitGeom s;
  SplitResult result = {};
  result.status = &act.header->status;
  if (g.chunks > 0 && plan_split(d, &s)) {
    int* n_parts = static_cast<int*>(workspace);
    uint32_t* most = static_cast<uint32_t*>(workspace) + 4;
    char* planes = static_cast<char*>(workspace) + split_head_bytes(s);
    partial = reinterpret_cast<float*>(planes + split_planes_bytes(s));
    result = {most, n_parts, s.slabs * s.grad_blocks, s.ctas, s.chunks, result.status};
    const cudaError_t e = launch_split(act, s, grad_out, planes, partial, most, stream);
    if (e != cudaSuccess) return e;
  }
  if (g.chunks > 65535 || (g.M + TM - 1) / TM > 65535) return cudaErrorNotSupported;
  if (g.chunks > 0) {
    dim3 grid(static_cast<unsigned>((g.N + TN - 1) / TN), static_cast<unsigned>((g.M + TM - 1) / TM),
              static_cast<unsigned>(g.chunks));
    auto launch = [&](auto kernel) {
      launch_kernel(kernel, grid, dim3(kThreads), 0, stream, result.most != nullptr, act.bitmap,
                    static_cast<const void*>(act.values), act.block_offsets, grad_out, partial, g, result);
    };
    auto launch_kind = [&](auto kind, auto span) {
      act.dt == 0 ? launch(dw_fp32_kernel<0, decltype(kind)::value, decltype(span)::value>)
                  : launch(dw_fp32_kernel<1, decltype(kind)::value, decltype(span)::value>);
    };
    using std::integral_constant;
    const bool span = g.tiles_per_img == 0;
    if (d.kind != 1) launch_kind(integral_constant<int, 0>{}, std::false_type{});
    else if (g.by_element) span ? launch_kind(integral_constant<int, 2>{}, std::true_type{})
                                : launch_kind(integral_constant<int, 2>{}, std::false_type{});
    else span ? launch_kind(integral_constant<int, 1>{}, std::true_type{})
              : launch_kind(integral_constant<int, 1>{}, std::false_type{});
    note_launches(1);
  }
  const long long mn = g.M * g.N;
  const int parts = result.most ? result.chunks : g.chunks;
  auto reduce = [&](auto kernel, int per_block, dim3 block) {
    launch_kernel(kernel, dim3(static_cast<unsigned>((mn + per_block - 1) / per_block)), block, 0, stream,
                  result.most != nullptr, partial, mn, g.chunks, result.n_parts, dw, accumulate, &act.header->status);
  };
  // Few outputs of many partial sums: eight threads each (432 of 96: 14 us by one thread each).
  if (parts >= 16 && mn < 65536) reduce(reduce_chunks_kernel<1, true>, 32, dim3(32, 8));
  else if (mn % 4 == 0 && mn >= 262144) reduce(reduce_chunks_kernel<4, false>, 1024, dim3(256));
  else reduce(reduce_chunks_kernel<1, false>, 256, dim3(256));
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace surgeon
