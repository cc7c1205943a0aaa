// Internal declarations shared by the translation units of libsurgeon (CUDA side only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "surgeon.h"

namespace surgeon {

// Storage type and magnitude-key mask per dtype.  The key is the bit pattern with the sign
// bit cleared, compared as an unsigned integer (Algorithm 1: prune step prunes by magnitude).
template <int DT> struct Elem;
template <> struct Elem<0> {
  using type = uint32_t;
  static constexpr uint32_t kKeyMask = 0x7FFFFFFFu;
  static constexpr uint32_t kSentinel = 0xFFFFFFFFu;
  static constexpr int kKeyBits = 31;
};
template <> struct Elem<1> {
  using type = uint16_t;
  static constexpr uint32_t kKeyMask = 0x7FFFu;
  static constexpr uint32_t kSentinel = 0xFFFFu;
  static constexpr int kKeyBits = 15;
};

constexpr int kBlockShift = 7;                       // log2(SURGEON_BLOCK)
constexpr int kBlockWords = SURGEON_BLOCK / 32;      // bitmap words per offset block
static_assert((1 << kBlockShift) == SURGEON_BLOCK, "SURGEON_BLOCK must be 128");

// ---- scratch of surgeon_prune_compact ---------------------------------------------------------
// Compaction tile ("chunk") = 4 KB of input = 256 16-byte vectors: the unit one warp works on and
// the unit of the exclusive scan that places it.
constexpr int kTileVecs = 256;
constexpr int64_t compact_tile_elems(int dt) { return dt == 0 ? 1024 : 2048; }
constexpr int kSelBinsLog2 = 9;        // bins of the select's histograms, over the bracket's keys
constexpr int kSelBins = 1 << kSelBinsLog2;
constexpr int kSelHists = 8;           // rounds of the select (2 in the common case)
constexpr int kSampleBins = 16384;     // bins of the sample
constexpr int kSelPhases = 12;         // grid-wide exchanges of a call (3 in the common case)
constexpr int kSelMaxCtas = 256;
constexpr int kClaimSets = 4, kClaimStride = 32;
__host__ __device__ constexpr int table_bins(int dt) { return dt == 0 ? 1 : 256; }       // whose counts every CTA shows to the others
__host__ __device__ constexpr size_t table_entries(int64_t chunks, int dt) {             // (a CTA has 16 chunks or all)
  return static_cast<size_t>(chunks / 16 + 1 < kSelMaxCtas ? chunks / 16 + 1 : kSelMaxCtas) * table_bins(dt);
}
// Candidate slots: per chunk, room for 1/16 of its elements (fp32: 32-bit keys, bf16: 16-bit).
__host__ __device__ constexpr int slot_entries(int dt) { return dt == 0 ? 64 : 128; }
constexpr int slot_entry_bytes(int dt) { return dt == 0 ? 4 : 2; }

// Byte offsets of the parts of the scratch buffer; nothing in it has to start at any value.
// arrive / answer / keys: what the CTAs exchange; hist: the select's histograms, one per round; claims:
// counters of claimed chunks; cnt
// and prefix: per-chunk counts and places of CTAs with too many chunks for shared memory; table: per CTA (16 chunks or more
// of a tensor) the counts of its bins; slots: the keys inside the bracket, per chunk.
struct PruneLayout {
  size_t arrive, answer, keys, hist, claims, cnt, prefix, table, slots, total;
  int64_t tiles;
};
constexpr PruneLayout prune_layout(int64_t n, int dt) {
  PruneLayout L{};
  L.tiles = (n + compact_tile_elems(dt) - 1) / compact_tile_elems(dt);
  const size_t t = static_cast<size_t>(L.tiles);
  size_t off = 0;
  L.arrive = off; off += static_cast<size_t>(kSelPhases) * kSelMaxCtas * 16;
  L.answer = off; off += static_cast<size_t>(kSelPhases) * (kSelMaxCtas + 2) * 16;
  L.keys = off; off += static_cast<size_t>(kSelMaxCtas) * 64 * 4;
  L.hist = off; off += static_cast<size_t>(kSelHists) * kSelBins * 4;
  L.claims = off; off += static_cast<size_t>(kSelPhases) * kClaimSets * kClaimStride * 4;
  L.prefix = off; off += t * 8;
  L.cnt = off; off += t * 4;
  off = (off + 255) & ~static_cast<size_t>(255);
  L.table = off;
  off += table_entries(L.tiles, dt) * 16;
  L.slots = off;
  off += t * static_cast<size_t>(slot_entries(dt)) * slot_entry_bytes(dt);
  L.total = (off + 255) & ~static_cast<size_t>(255);
  return L;
}
constexpr size_t prune_workspace_bytes(int64_t n, int dt) { return prune_layout(n, dt).total; }

// Host launchers (each enqueues on `stream` and returns the last CUDA error).
cudaError_t launch_prune_compact(const void* x, int64_t n, int dt, int64_t k,
                                 const surgeon_compressed& out, void* workspace,
                                 cudaStream_t stream, int drop_zeros = 0, int stall = 0, int share = 0);
cudaError_t launch_decompress(const surgeon_compressed& act, void* x_out, cudaStream_t stream);
// Eq. 4 on device: *gi_out = sqrt(sum dw^2 / n); workspace = SURGEON_GI_WORKSPACE_BYTES of scratch.
cudaError_t launch_gradient_importance(const float* dw, long long n, double* gi_out,
                                       void* workspace, cudaStream_t stream);

size_t weight_grad_fp32_workspace(const surgeon_layer_desc& d);
cudaError_t launch_weight_grad_fp32(const surgeon_compressed& act, const surgeon_layer_desc& d,
                                    const float* grad_out, float* dw, int accumulate,
                                    void* workspace, cudaStream_t stream);

size_t weight_grad_grouped_workspace(const surgeon_layer_desc& d);
cudaError_t launch_weight_grad_grouped(const surgeon_compressed& act, const surgeon_layer_desc& d,
                                       const float* grad_out, float* dw, int accumulate,
                                       void* workspace, cudaStream_t stream);

size_t weight_grad_tc_workspace(const surgeon_layer_desc& d);
cudaError_t launch_weight_grad_tc(const surgeon_compressed& act, const surgeon_layer_desc& d,
                                  const float* grad_out, float* dw, int accumulate, int share,
                                  void* workspace, cudaStream_t stream);

// The driver's cuTensorMapEncodeTiled, looked up through the runtime (the library carries no
// link-time dependency on the driver library); nullptr if unavailable.
void* tensor_map_encode_fn();
// Number of SMs of the current device (cached per device id).
int sm_count();
// Lets `kernel` use `bytes` of dynamic shared memory; the attribute is set when a kernel first
// needs that much on a device, later calls only look it up.
cudaError_t allow_dynamic_smem(const void* kernel, int bytes);
// Adds to the process-wide kernel-launch counter behind surgeon_launch_count().
void note_launches(int n);

// Programmatic dependent launch.  A kernel launched with `dependent` set may start while the
// kernel before it on the stream is still running (once every CTA of that kernel has called
// pdl_trigger or has exited): its set-up then overlaps the predecessor's tail.  It must call
// pdl_wait before it touches anything the predecessor writes; pdl_wait returns when the
// predecessor has completed and its writes are visible.  Both calls do nothing in a kernel that
// was launched the ordinary way.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// The first kernel of a weight-gradient call: it waits for what came before on the stream, zeroes the
// call's status word (a memset of its own cost 2 us of host time and as much of the stream's), and
// only then lets its dependents start, which read the store without waiting for anything else.
__device__ __forceinline__ void prepass_begin(uint32_t* status) {
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) { *status = 0u; __threadfence(); }
  pdl_trigger();
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                 cudaStream_t stream, bool dependent, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Checked builds (-DSURGEON_BOUNDS, the library's stand-in for a memory checker): every guarded
// global store tests its index against the size the host computed for the buffer; an index
// outside records SURGEON_ERR_INTERNAL in `status_word` and the store is skipped.  In the
// ordinary build the test compiles away.
#ifdef SURGEON_BOUNDS
#define SURGEON_IN_BOUNDS(idx, limit, status_word)                                              \
  ((static_cast<unsigned long long>(idx) < static_cast<unsigned long long>(limit)) ||           \
   (atomicMax((status_word), static_cast<uint32_t>(SURGEON_ERR_INTERNAL)), false))
#else
#define SURGEON_IN_BOUNDS(idx, limit, status_word) true
#endif

// Division of numbers below 2^31 by one that the host knows: two instructions instead of some 35 (Granlund and Montgomery,
// "Division by invariant integers using multiplication", 1994).
struct FastDiv {
  uint32_t mul, shift;
};
inline FastDiv make_div(uint32_t d) {            // d >= 1
  FastDiv f{0, 0};
  while ((1ull << f.shift) < d) ++f.shift;
  f.mul = static_cast<uint32_t>(((1ull << 32) * ((1ull << f.shift) - d)) / d + 1);
  return f;
}
__device__ __forceinline__ uint32_t divide(uint32_t n, FastDiv f) { return (__umulhi(n, f.mul) + n) >> f.shift; }

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}
__device__ __forceinline__ uint32_t warp_sum(uint32_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}
// Exclusive prefix sum over the lanes of a warp.
__device__ __forceinline__ uint32_t warp_excl_scan(uint32_t v) {
  uint32_t s = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(0xFFFFFFFFu, s, o);
    if (lane_id() >= static_cast<uint32_t>(o)) s += t;
  }
  return s - v;
}

}  // namespace surgeon
