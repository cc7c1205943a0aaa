// The fp32 path of surgeon_weight_grad on the tensor cores (weight_grad_fp32_split.cu), as the path's launcher
// (weight_grad_fp32.cu) uses it.
#pragma once

#include "surgeon_internal.cuh"

namespace surgeon {

// Both operands are multiplied by 2^24 before they are cut: a subnormal number's last bit, 2^-149, then is 2^-125, so the
// parts of every number are normal bf16 numbers, and a product that is lost (below 2^-126) is below 2^-174, of which
// an fp32 sum keeps nothing.  The partial sums carry the factor of both operands, 2^48.
constexpr int kSplitShift = 24;
constexpr int kSplitTileK = 64;

struct SplitGeom {
  int C, H, W, O, KW, RS, stride, pad, OH, OW;
  int P, K, N;              // positions per image (linear: 1), what the GEMM sums over, its columns (c, r, s)
  int step_y, step_x;       // 64 positions, in rows and columns of the output
  int most_len;             // positions of one output row that 32 input elements hold
  int linear, vec;          // vec: the gradient can be read 16 bytes at a time
  int grad_blocks;          // blocks of the pre-pass that writes the gradient's planes
  uint32_t n_words;         // words of the bitmap
  FastDiv by_p, by_ow;      // division by P and OW
  int tile_n, nt, mt;       // output channels per CTA, tiles of them, tiles of 128 columns
  int warp_cols, tmem_cols;
  int k_tiles, per_chunk, chunks, ctas;
  int slabs, slab_chunks;   // the chunks are taken so many at a time, so that the gradient's planes stay small
  int kt0, chunk0;          // (set for each launch) the slab's first K-tile and chunk
  uint32_t* status;         // (likewise) the store's status word, for checked builds
};
// False: the layer is not one for it.
bool plan_split(const surgeon_layer_desc& d, SplitGeom* out);
__host__ __device__ __forceinline__ int slab_tiles(const SplitGeom& g) {        // K-tiles of the slab from kt0 on
  const int all = g.slab_chunks * g.per_chunk, left = g.k_tiles - g.kt0;
  return all < left ? all : left;
}
__host__ __device__ __forceinline__ size_t split_planes_bytes(const SplitGeom& g) {      // of that slab; the first one's are the most
  return static_cast<size_t>(slab_tiles(g)) * g.nt * 3 * g.tile_n * kSplitTileK * 2;
}
// partial: [chunks][O][N].  most: the largest magnitudes of the gradient (a word per block of the pre-passes) and then of the
// activation (a word per CTA), as bf16 patterns of the scaled numbers; 0xFFFF from a CTA that gave up.
cudaError_t launch_split(const surgeon_compressed& act, const SplitGeom& g, const float* grad_out, void* planes,
                         float* partial, uint32_t* most, cudaStream_t stream);

}  // namespace surgeon
