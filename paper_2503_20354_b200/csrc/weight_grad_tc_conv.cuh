// Plans and launchers of the tensor-core weight-gradient kernels, and the gradient pre-passes (weight_grad_tc_conv.cu).
#pragma once

#include <cuda.h>

#include "surgeon_internal.cuh"

#include <cstring>

namespace surgeon {

// Plans depend only on the layer geometry (and the device's SM count): a weight-gradient call
// looks its plan up in a small per-thread table instead of searching tilings and split counts
// again (the searches cost microseconds, as much as a kernel launch).  `Tag` separates the tables
// of the different planners.
template <typename Tag, typename P, typename F>
inline bool memo_plan(const surgeon_layer_desc& d, int extra, P* out, F compute) {
  struct Entry { surgeon_layer_desc d; int extra, dev; bool used, ok; P p; };
  constexpr int kEntries = 128;                  // (a layer has up to two plans)
  thread_local Entry table[kEntries] = {};
  thread_local int next = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
  for (int i = 0; i < kEntries; ++i) {
    const Entry& e = table[i];
    if (e.used && e.extra == extra && e.dev == dev && std::memcmp(&e.d, &d, sizeof(d)) == 0) {
      if (e.ok) *out = e.p;
      return e.ok;
    }
  }
  Entry& e = table[next];
  next = (next + 1) % kEntries;
  e.d = d; e.extra = extra; e.dev = dev; e.used = true;
  e.p = P{};
  e.ok = compute(&e.p);
  if (e.ok) *out = e.p;
  return e.ok;
}

// fp32 -> bf16 (round to nearest even) copy of n elements, as one streaming kernel.
// As every gradient pre-pass, it also zeroes the call's status word.
cudaError_t launch_grad_to_bf16(const float* g, long long n, void* out_bf16, uint32_t* status, cudaStream_t stream);
// The same for `rows` rows of `len` elements, written with a row pitch of `pitch` >= len
// elements (a multiple of 8); the padding is zero.
cudaError_t launch_grad_to_bf16_rows(const float* g, long long rows, int len, int pitch,
                                     void* out_bf16, uint32_t* status, cudaStream_t stream);

// ---- convolutions whose operand has to be expanded (weight_grad_tc_strided.cu) -----------------
struct StridedParams {
  int B, C, H, W, O, KH, KW, stride, pad, OH, OW;
  int OWp, P;               // output row padded to a multiple of 8 positions; positions per image (OH * OWp)
  int RS, n_gemm;           // KH * KW, C * RS
  int acc_n, n_acc;         // columns per accumulator, accumulators per CTA (1 or 2)
  int m_tiles, n_tiles, splits;
  int rows_per_tile;        // im2col rows per CTA (a multiple of 8, at most 128 m_acc)
  int m_acc, a_bytes;       // row tiles of a CTA (1 or 2), operand bytes of a stage
  int tiles_per_img;        // K-tiles of 64 positions
  int macro;                // K-tiles per rebuilt patch
  int macros_per_img, total_macros, macros_per_split;
  int patch_rows, plane, row_len;    // input rows of a patch, elements of a phase plane of one row, of a row with its padding
  int patch_bytes, stages, tmem_cols, smem_bytes;
  unsigned inv_stride;      // ix / stride = ix * inv_stride >> 16
  FastDiv by_row, by_ch;    // division by the pieces per row, and per channel of the patch,
  FastDiv by_owp, by_macros;         // by OWp, and by the macros of an image,
  FastDiv by_rs, by_kw, by_stride;   // by RS, KW and the stride
  unsigned partial_blk;     // index of the bitmap's last block if it is partial, else 0xFFFFFFFF (launcher)
  long long n_words;        // words of the bitmap (filled by the launcher)
};
bool plan_strided(const surgeon_layer_desc& d, StridedParams* out);
size_t strided_partial_bytes(const StridedParams& p);
size_t strided_grad_bf16_bytes(const StridedParams& p);
// partial = [splits][O][n_gemm] fp32, status = one word (the pre-pass zeroes it).
cudaError_t launch_strided(const surgeon_compressed& act, const StridedParams& p, const float* grad_out,
                           void* grad_bf16, float* partial, uint32_t* status, cudaStream_t stream);

// ---- layers whose im2col operand is the activation itself (weight_grad_tc_direct.cu) ----------
struct DirectParams {
  int mode;                 // 0 = linear [T, C] (MN-major operands), 1 = conv 1x1 stride 1 (K-major),
                            // 2 = conv 1x1 stride 2 (K-major, sampled input), 3 = the same on a transposed gradient copy
  int ow, in_w, in_hw;      // mode 2: output row length, input row length, input plane size
  int taps;                 // 1, or kh*kw for a k x k stride-1 conv (mode 1 over shifted gradients)
  int kh, kw, pad, in_h, oh;  // taps > 1: kernel and map sizes (with ow, in_w)
  int o_real;               // output channels of the layer; O = taps * o_real
  int row_shift;            // taps > 1: only the kw column shifts are stored; rows shift by TMA offset
  int tg;                   // k x k on one transposed gradient copy: 1-5 (see weight_grad_tc_direct.cu), else 0
  int map_rows, kpos;       // tg: whole map rows per K-tile, and their positions
  int slot_w;               // mode 3: K positions per output row: 8, 16, 32 or 64
  unsigned many_keep;       // mode 3: packed values above which a warp's lanes share each run (launcher)
  int k_rows;               // tg: k-rows of a 64-channel slab in shared memory
  int unit_bytes, b_bytes;  // tg: bytes of a unit's slabs, and of a stage
  unsigned box_bytes;       // tg: bytes one box brings
  int copies;               // stacked gradient copies: taps, or kw with row_shift
  int g_len;                // conv: elements per row of the gradient copy (T, or oh * in_w)
  int upt, n_units;         // conv: accumulator units per tap (of acc_n columns), units in all
  int C, O;                 // input channels / gradient channels (taps * output channels)
  int T;                    // linear: rows; conv: positions per image
  int pitch;                // elements per row of the bf16 gradient copy
  int imgs;                 // conv: batch; linear: 1
  int acc_n, n_acc, n_cols; // columns per accumulator, accumulators per CTA, their product
  int m_tiles, n_tiles, splits;
  int tiles_per_img, total_ktiles, ktiles_per_split;
  int rows_per_tile;        // channels per row tile (128, or fewer when C is spread evenly; a multiple of 16)
  int pair;                 // 1: CTA pairs (cta_group::2) over two row tiles; m_tiles is then even
  int a_stages, b_stages;   // depth of the activation-tile and gradient-tile rings
  int tmem_cols, smem_bytes;
  long long n_words;        // words of the bitmap (filled by the launcher)
  const long long* n_keep_ptr;  // device address of the store's count of packed values (launcher)
  unsigned few_keep;        // packed values up to which runs are rebuilt element by element (launcher)
  unsigned partial_blk;     // index of the bitmap's last block if it is partial, else 0xFFFFFFFF
};
bool plan_direct(const surgeon_layer_desc& d, bool share, DirectParams* out);   // share: other streams' calls run beside it
bool plan_direct_copies(const surgeon_layer_desc& d, DirectParams* out);   // never a transposed gradient copy
size_t direct_grad_bf16_bytes(const DirectParams& p);
// partial = [splits][O][C] fp32 (O counts the stacked taps), status = one word (the pre-pass zeroes it).
cudaError_t launch_direct(const surgeon_compressed& act, const DirectParams& p,
                          const float* grad_out, void* grad_bf16, float* partial,
                          uint32_t* status, cudaStream_t stream);
// The pre-pass that writes the bf16 copy (or shifted copies) of the output gradient, and the
// tensor map over it (conv: boxes of 64 positions x box_rows rows; linear: 64 columns x 64 rows).
cudaError_t launch_direct_prepass(const DirectParams& p, const float* grad_out, void* grad_bf16,
                                  uint32_t* status, cudaStream_t stream);
cudaError_t encode_direct_grad_map(const DirectParams& p, void* grad_bf16, int box_rows, CUtensorMap* out);

// ---- the same layers on CTA pairs with the operand roles exchanged (weight_grad_tc_swap.cu) -----
struct SwapParams {
  DirectParams d;           // layer geometry and the layout of the bf16 gradient copy
  int nt, half;             // input channels per pair tile (MMA N, a multiple of 16) and per CTA
  int n_acc;                // accumulators per CTA: 128 gradient rows x nt channels each
  int lpr;                  // lanes (runs of 32 elements) per row of the activation tile: 2 or 4
  // conv: the stacked gradient rows (tap, output channel) are cut into units of 128 TMEM lanes.
  // Per tap a_units full units of 128 rows (one TMA box each; the last may be partly filled when
  // rem_box is 0); the o_real - 128 * a_full rows left over, if any, go `rpu` taps to a unit in
  // boxes of rem_box rows (a power of two below 128).
  int a_full, a_units, rem_box, rpu;
  int n_units;              // units in all (linear: groups of 128 gradient columns)
  int m_tiles, n_tiles, splits, ktiles_per_split;
  int gw, groups;           // warps per producer group, groups (one K-tile in flight per group)
  int a_stages, g_stages;   // depth of the activation-tile and gradient-tile rings
  int stage_bytes;          // staging area of packed values (fp32 activations), 0 if none
  int tmem_cols, smem_bytes;
  long long n_words;        // words of the bitmap (filled by the launcher)
  const long long* n_keep_ptr;
  unsigned partial_blk;     // index of the bitmap's last block if it is partial, else 0xFFFFFFFF
};
bool plan_swap(const surgeon_layer_desc& d, SwapParams* out);
int swap_resident_pairs();   // CTA pairs the device holds at once
size_t swap_partial_bytes(const SwapParams& p);
// partial = [splits][O][C] fp32 (O counts the stacked taps), status = one word (the pre-pass zeroes it).
cudaError_t launch_swap(const surgeon_compressed& act, const SwapParams& p, const float* grad_out,
                        void* grad_bf16, float* partial, uint32_t* status, cudaStream_t stream);

}  // namespace surgeon
