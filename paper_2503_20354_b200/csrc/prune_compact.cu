// Threshold select and compaction of surgeon_prune_compact, and surgeon_decompress.
//
// Algorithm 1, prune step: the kept set of a layer is its n_keep largest-magnitude elements, ties
// at the threshold broken by lowest flat index.  Its decompose step / Section 4.2: the pruned
// activation is cached as the vector of kept elements plus one index bit per element.
//
// One cooperative kernel does the whole call: every CTA owns a contiguous range of 4 KB chunks
// (the unit one warp works on, fetched by TMA into a ring of its own), and the CTAs meet at two or
// three grid-wide exchanges, at which CTA 0 collects, decides and answers:
//
//   sample    a scattered sample gives a bracket [lo, hi] of keys that contains the threshold with
//             overwhelming probability (1-4 % of the elements)
//   classify  first pass over the CTA's chunks: keys above the bracket are counted per chunk, the
//             keys inside are listed and counted in a histogram of 512 bins over the bracket
//   exchange  the summed histogram gives the threshold's bin: one key for bf16, whose brackets are
//             narrower than 512 keys, some thousands of keys for fp32, of which few occur
//   exchange  every CTA reports its count above the bin and the keys it has inside; CTA 0 finds the
//             threshold among them and gives every CTA its place in the packed vector
//   emit      the lists complete the per-chunk counts, a scan turns them into places, and a second
//             pass over the chunks, last one first, writes the store
//
// Why one kernel: as four kernels behind a memset a call took 45-60 us whatever the tensor's size,
// most of it launches, drained pipelines and grids that started empty; an exchange costs about 2 us.
// A tensor of at most 48 chunks per SM (29 MB) stays in shared memory between the passes, so it is
// read from memory once; of a larger one the end of each CTA's range stays, and the second pass
// starts there and goes backwards, where the L2 cache still holds most of what it needs.
//
// When the sample misleads (the bracket misses, or holds more equal keys than a list takes) the
// first pass is repeated with the bracket the counts prove; the result is exact and unique
// either way.  Every count fits 32 bits because n <= SURGEON_MAX_N < 2^31.
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <random>

#include "surgeon_internal.cuh"
#include "tc_common.cuh"

namespace surgeon {

namespace {

using tc::smem_u32;

constexpr uint32_t kFull = 0xFFFFFFFFu;

// ---- geometry -----------------------------------------------------------------------------------
// A chunk is 32 rows of 128 bytes (128-byte swizzle, so that 32 lanes can each read their own row
// without bank conflicts): each LANE owns one row, i.e. 32 (fp32) or 64 (bf16) consecutive
// elements, and bitmap words are built without cross-lane traffic.
constexpr int kWarps = 16;                       // one CTA per SM; 128 registers a thread
constexpr int kThreads = kWarps * 32;
constexpr int kSlotsPerWarp = 3;                 // chunks in flight per warp: 192 KB per SM
constexpr int kChunkBytes = 4096;
constexpr int kRingBytes = kWarps * kSlotsPerWarp * kChunkBytes;
constexpr int kResidentChunks = kWarps * kSlotsPerWarp;
// The rest of the shared memory.  Slots: the listed keys, room for 1/16 of every chunk.
constexpr int kMaxLocalChunks = 1024;            // per-chunk counts in shared memory up to here
constexpr int kSlotBytes = 256;
constexpr int kAuxSlots = 8192;                  // (histograms before it)
constexpr int kAuxCnt = kAuxSlots + kResidentChunks * kSlotBytes;
constexpr int kAuxPrefix = kAuxCnt + kMaxLocalChunks * 4;
constexpr int kSampleBinsLog2 = 14;              // top 14 key bits: 64 bins per octave; 16-bit counters here
constexpr int kSampleBytes = 2 << kSampleBinsLog2;
static_assert((1 << kSampleBinsLog2) == kSampleBins, "bins of the sample");
constexpr int kAuxBytes = kAuxPrefix + kMaxLocalChunks * 8 > kSampleBytes ? kAuxPrefix + kMaxLocalChunks * 8 : kSampleBytes;
// emit: per-warp staging of the kept values of a sparse chunk, in the place of histogram and slots
constexpr int kStageBytes = (kAuxCnt / kWarps) & ~15;
constexpr size_t kPruneSmem = static_cast<size_t>(kRingBytes) + kAuxBytes + 1024;
static_assert(kChunkBytes == kTileVecs * 16, "chunk size");
// A streamed tensor's bracket comes from order statistics 2.5 sqrt(G) + 1 places to either side of the middle of G
// CTAs' answers: with fewer than 31 CTAs there are none, and every key would be a candidate.
constexpr int kLeastStreamedCtas = 31;
constexpr int kMaxKeys = 64;                     // keys one CTA reports at the last exchange
constexpr int kKeysPerThread = 8;                // and CTA 0 takes in
constexpr int kKeysAtOnce = kKeysPerThread * kThreads;

struct PruneArgs {
  const void* x;
  long long n, n_rows_full;      // elements; whole 128-byte rows (what the tensor map covers)
  uint32_t k;
  int n_chunks;                  // chunks in all
  int drop_zeros, stall;
  int spread;                    // the chunks are claimed, and the counts are in global memory
  unsigned long long token;      // unlike any other call's
  surgeon_header* hdr;
  uint32_t* bitmap;
  void* values;
  uint32_t* offsets;
  ulonglong2* arrive;            // [kSelPhases][kSelMaxCtas]: {token, what the CTA reports}
  ulonglong2* answer;            // [kSelPhases][kSelMaxCtas + 2]: {token, what CTA 0 answers}
  uint32_t* keys;                // [kSelMaxCtas][kMaxKeys]
  uint32_t* hist;                // [kSelHists][kSelBins]
  uint32_t* claims;              // [kSelPhases][kClaimSets], kClaimStride words apart: groups claimed in each pass
  uint32_t* cnt;                 // per chunk (spread)
  unsigned long long* prefix;    // likewise
  void* slots;                   // per chunk, listed keys of ranges that are not resident
};

__device__ __forceinline__ uint32_t hash_u32(uint32_t v) {
  v ^= v >> 16; v *= 0x7FEB352Du; v ^= v >> 15; v *= 0x846CA68Bu; v ^= v >> 16;
  return v;
}

// ---- grid-wide exchange ----------------------------------------------------------------------------
// A CTA reports by storing {token, 8 bytes} in its own word of the phase; CTA 0 polls these words,
// one thread per CTA, and answers by storing {token, 8 bytes} in words that the others poll.  (Every
// CTA polling the words of all others took 4-6 us on 148 SMs: the same L2 lines, 148 times over.)
// No counter has to start at zero, so the call needs no memset: the token differs from call to
// call.  For a captured graph, whose replays carry the same token, CTA 0 clears every report that it
// has read, clears a phase's answers before it answers the phase before it, and clears the first
// answer (phase 0) after the reports of phase 1; a CTA that gives up takes its own words back.  All CTAs are
// resident (cooperative launch); polls are bounded.
__device__ __forceinline__ void word_store(ulonglong2* p, unsigned long long token, unsigned long long v) {
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}"
               ::"l"(p), "l"(token), "l"(v) : "memory");
}
__device__ __forceinline__ ulonglong2 word_load(const ulonglong2* p) {
  ulonglong2 v;
  asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
               : "=l"(v.x), "=l"(v.y) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// One thread waits for a word of this call (what it announces apart from its own 8 bytes is visible
// after a fence).  `stall` is the diagnostic of SURGEON_DEBUG_STALL_BARRIER: a value nobody ever
// stores, and a cap of 1024 polls.
__device__ __forceinline__ bool word_wait(const ulonglong2* p, unsigned long long token, unsigned long long* v,
                                          bool stall = false) {
  const uint32_t cap = stall ? 1024u : (1u << 22);
  for (uint32_t spins = 0; spins <= cap; ++spins) {
    const ulonglong2 w = word_load(p);
    if (w.x == (stall ? ~token : token)) {
      *v = w.y;
      return true;
    }
    if (spins > 64u) __nanosleep(20);
  }
  return false;
}

// bf16 keys are compared two at a time inside their 32-bit word: a key is at most 0x7FFF, so
// key + (0x8000 - t) carries into bit 15 of its half exactly when key >= t, and never into the
// other half.  The flag bits of the 16 words of a group of 32 elements are collected in one mask,
// word i shifted right by i: bit (15 - i) is element 2i, bit (31 - i) element 2i + 1.
__device__ __forceinline__ uint32_t ge_const(uint32_t t) {       // t in [0, 0x8000]
  return (0x8000u - (t > 0x8000u ? 0x8000u : t)) * 0x10001u;
}
__device__ __forceinline__ uint32_t pair_flags(uint32_t keys2, uint32_t c, int i) {
  return ((keys2 + c) >> i) & (0x80008000u >> i);
}
// The same mask in element order (bit e = element e).
__device__ __forceinline__ uint32_t pairs_to_element_order(uint32_t m) {
  const uint32_t r = __brev(m);              // bit (16 + i): element 2i, bit i: element 2i + 1
  auto spread = [](uint32_t x) {             // bit i -> bit 2i, for x < 2^16
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
  };
  return spread(r >> 16) | (spread(r & 0xFFFFu) << 1);
}
__device__ __forceinline__ uint32_t valid_mask(int nv, int w) {
  const int left = nv - 32 * w;
  return left >= 32 ? 0xFFFFFFFFu : (left <= 0 ? 0u : ((1u << left) - 1u));
}

// This lane's row (8 vectors) out of the swizzled chunk.
__device__ __forceinline__ void load_row(const unsigned char* region, uint4 (&q)[8]) {
  const uint32_t lane = lane_id();
  const unsigned char* row = region + lane * 128;
#pragma unroll
  for (int j = 0; j < 8; ++j) q[j] = *reinterpret_cast<const uint4*>(row + ((j ^ (lane & 7)) << 4));
}
// Element e of this lane's row.
template <int DT>
__device__ __forceinline__ uint32_t row_elem(const unsigned char* region, int e) {
  using E = typename Elem<DT>::type;
  const uint32_t lane = lane_id();
  const int byte = e * static_cast<int>(sizeof(E));
  return static_cast<uint32_t>(*reinterpret_cast<const E*>(region + lane * 128 + (((byte >> 4) ^ (lane & 7)) << 4) + (byte & 15)));
}

// Masks of the elements with key >= t, bit e = element e, elements past nv cleared.  fp32 keys are
// below 2^31, so the sign bit of (key - t) says key < t; a funnel shift collects it (two
// instructions per element), element e in bit 31 - e, and one bit reversal puts it back.
template <int DT, int WPL>
__device__ __forceinline__ void mask_ge(const uint4 (&q)[8], int nv, uint32_t t, uint32_t (&m)[WPL]) {
  const uint32_t c_t = ge_const(t);
#pragma unroll
  for (int w = 0; w < WPL; ++w) m[w] = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t c[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int pw = 4 * j + i;
      if (DT == 0) m[0] = __funnelshift_l((c[i] & Elem<DT>::kKeyMask) - t, m[0], 1);
      else m[(pw >> 4) % WPL] |= pair_flags(c[i] & 0x7FFF7FFFu, c_t, pw & 15);
    }
  }
#pragma unroll
  for (int w = 0; w < WPL; ++w)
    m[w] = (DT == 0 ? ~__brev(m[w]) : pairs_to_element_order(m[w])) & valid_mask(nv, w);
}

// The chunk's keys inside the bracket (flagged in cw0 / cw1, `c_tot` of them in the warp) if they
// all are one key, else 0 (no key inside a bracket is 0).  Called where massive ties overflow a
// list, and kept out of line so that the first pass's registers are those of its common path.
template <int DT>
__device__ __noinline__ uint32_t one_key_of_chunk(const unsigned char* region, uint32_t cw0, uint32_t cw1,
                                                  uint32_t c_tot) {
  constexpr uint32_t kMask = Elem<DT>::kKeyMask;
  const uint32_t lane = lane_id();
  const unsigned char* row = region + lane * 128;
  const int src = __ffs(__ballot_sync(kFull, (cw0 | cw1) != 0u)) - 1;
  uint32_t k0 = 0;
  if (static_cast<int>(lane) == src)                                   // (fp32: cw1 is cw0)
    k0 = row_elem<DT>(region, cw0 ? __ffs(cw0) - 1 : 32 + __ffs(cw1) - 1) & kMask;
  k0 = __shfl_sync(kFull, k0, src);
  uint32_t eq = 0;
  const uint32_t c_ge = ge_const(k0), c_gt = ge_const(k0 + 1u);
#pragma unroll 1
  for (int j = 0; j < 8; ++j) {                  // one 16-byte piece at a time: few registers
    const uint4 v = *reinterpret_cast<const uint4*>(row + ((j ^ (lane & 7)) << 4));
    const uint32_t c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (DT == 0) {
        eq += (c[i] & kMask) == k0 ? 1u : 0u;
      } else {
        const uint32_t keys2 = c[i] & 0x7FFF7FFFu;
        eq += __popc(((keys2 + c_ge) & ~(keys2 + c_gt)) & 0x80008000u);
      }
    }
  }
  // (rows past the tensor's end hold key 0)
  return __reduce_add_sync(kFull, eq) == c_tot ? k0 : 0u;
}

// Keep only the lowest `allowed` set bits of `m`.
__device__ __forceinline__ uint32_t lowest_set_bits(uint32_t m, long long allowed) {
  if (allowed <= 0) return 0u;
  int extra = __popc(m) - static_cast<int>(allowed < 32 ? allowed : 32);
  while (extra > 0) {
    m &= ~(0x80000000u >> __clz(m));
    --extra;
  }
  return m;
}

__device__ __forceinline__ unsigned long long warp_incl_u64(unsigned long long v) {
  const uint32_t lane = lane_id();
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long up = __shfl_up_sync(kFull, v, o);
    if (lane >= static_cast<uint32_t>(o)) v += up;
  }
  return v;
}

// ---- emit one chunk -------------------------------------------------------------------------------
// before = (elements above the threshold before the chunk) << 32 | (ties before it); n_eq = its ties.
// True when the chunk's place in the ring has been written to.
template <int DT>
__device__ __forceinline__ bool emit_chunk(const PruneArgs& a, unsigned char* region, unsigned char* stage,
                                           int chunk, uint32_t tau, long long quota,
                                           unsigned long long before, uint32_t n_eq, long long n_stored) {
  using E = typename Elem<DT>::type;
  constexpr int EPR = 128 / sizeof(E);         // elements per row (= per lane): 32 / 64
  constexpr int EPV = 16 / sizeof(E);          // elements per 16-byte vector: 4 / 8
  constexpr int WPL = EPR / 32;                // bitmap words per lane: 1 / 2
  constexpr int BPC = 32 * EPR / SURGEON_BLOCK;   // offset blocks per chunk: 8 / 16
  constexpr int LPB = 32 / BPC;                // lanes per offset block: 4 / 2
  const uint32_t lane = lane_id();
  E* __restrict__ values = reinterpret_cast<E*>(a.values);
  uint4 q[8];
  load_row(region, q);
  const long long grow = static_cast<long long>(chunk) * 32 + lane;   // row index in the tensor
  long long left = a.n - grow * EPR;
  const int nv = left < 0 ? 0 : (left > EPR ? EPR : static_cast<int>(left));
  const long long eq_b = static_cast<long long>(before & 0xFFFFFFFFull);
  const long long eq_e = eq_b + n_eq;
  // every tie of the chunk is kept, or none is; in the one chunk inside which the quota ends they
  // are ranked by flat index (= lane, then bit)
  const bool ties = eq_e <= quota;
  uint32_t word[WPL];
  mask_ge<DT, WPL>(q, nv, ties ? tau : tau + 1u, word);
  if (!ties && eq_b < quota) {
    uint32_t ge[WPL], ec = 0;
    mask_ge<DT, WPL>(q, nv, tau, ge);
#pragma unroll
    for (int w = 0; w < WPL; ++w) { ge[w] &= ~word[w]; ec += __popc(ge[w]); }
    long long allowed = quota - eq_b - warp_excl_scan(ec);
#pragma unroll
    for (int w = 0; w < WPL; ++w) {
      word[w] |= lowest_set_bits(ge[w], allowed);
      allowed -= __popc(ge[w]);
    }
  }
  uint32_t cnt = 0;
#pragma unroll
  for (int w = 0; w < WPL; ++w) cnt += __popc(word[w]);
  uint32_t incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t up = __shfl_up_sync(kFull, incl, o);
    if (lane >= static_cast<uint32_t>(o)) incl += up;
  }
  const uint32_t lane_pre = incl - cnt;
  const uint32_t total = __shfl_sync(kFull, incl, 31);
  const long long kept_before = static_cast<long long>(before >> 32) + (eq_b < quota ? eq_b : quota);

  // ---- bitmap words and block offsets: coalesced ----
  const long long n_words = (a.n + 31) / 32;
  const long long n_blocks = (a.n + SURGEON_BLOCK - 1) >> kBlockShift;
  const long long wi = static_cast<long long>(chunk) * 32 * WPL + lane * WPL;
  if (WPL == 2 && wi + 1 < n_words) {
    *reinterpret_cast<uint2*>(a.bitmap + wi) = make_uint2(word[0], word[WPL - 1]);
  } else if (wi < n_words) {
    a.bitmap[wi] = word[0];
  }
  const uint32_t off = __shfl_sync(kFull, lane_pre, (lane * LPB) & 31);
  const long long blk = static_cast<long long>(chunk) * BPC + lane;
  if (lane < BPC && blk < n_blocks) a.offsets[blk] = static_cast<uint32_t>(kept_before) + off;
  if (total == 0) return false;

  // ---- kept values, in packed order into shared memory, then out as 16-byte vectors ----
  // The sequence starts `mis` elements into its place, mis = the misalignment of its destination in
  // `values`: 16-byte vectors of the two then line up.
  const uint32_t mis = static_cast<uint32_t>(kept_before % EPV);
  const uint32_t most = __reduce_max_sync(kFull, cnt);
  // Sparse rows: a loop over the set bits, which fetches each kept element from the row; its cost is
  // that of the fullest row (about 13 instructions per element), the unrolled gather's is 5 per element
  // of the row, kept or not.
  const bool sparse = most <= (DT == 0 ? 12u : 26u) &&
                      (total + mis) * sizeof(E) <= static_cast<uint32_t>(kStageBytes);
  if (sparse) {
    uint32_t sa = smem_u32(stage) + (lane_pre + mis) * static_cast<uint32_t>(sizeof(E));
#pragma unroll
    for (int w = 0; w < WPL; ++w) {
      uint32_t m = word[w];
      while (m) {
        const int e = 32 * w + __ffs(m) - 1;
        m &= m - 1;
        const uint32_t v = row_elem<DT>(region, e);
        if (DT == 0) asm volatile("st.shared.u32 [%0], %1;" ::"r"(sa), "r"(v) : "memory");
        else asm volatile("st.shared.u16 [%0], %1;" ::"r"(sa), "h"(static_cast<unsigned short>(v)) : "memory");
        sa += static_cast<uint32_t>(sizeof(E));
      }
    }
    __syncwarp();
    const E* outp = reinterpret_cast<const E*>(stage);
    E* gbase = values + (kept_before - mis);
    const uint32_t end = mis + total, v_first = mis ? 1u : 0u, v_end = end / EPV;
    if (mis) {
      const uint32_t sl = mis + lane;
      if (sl < static_cast<uint32_t>(EPV) && sl < end &&
          SURGEON_IN_BOUNDS(kept_before - mis + sl, n_stored, &a.hdr->status))
        gbase[sl] = outp[sl];
    }
    for (uint32_t g = v_first + lane; g < v_end; g += 32)
      if (SURGEON_IN_BOUNDS(kept_before - mis + g * EPV + EPV - 1, n_stored, &a.hdr->status))
        *reinterpret_cast<uint4*>(gbase + g * EPV) = *reinterpret_cast<const uint4*>(stage + g * 16);
    const uint32_t t0 = (v_end > v_first ? v_end : v_first) * EPV;
    if (t0 + lane < end && SURGEON_IN_BOUNDS(kept_before - mis + t0 + lane, n_stored, &a.hdr->status))
      gbase[t0 + lane] = outp[t0 + lane];
    __syncwarp();                                // the staging area is this warp's next chunk's
    return false;
  }
  // Dense rows: gathered in place in the chunk's own part of the ring.
  __syncwarp();                                  // every lane has its row in registers
  // The byte at address a of the packed sequence lives at a ^ ((a >> 5) & 0x7C): the 32-bit word
  // index is XORed with the index of its 128-byte row.  Without it, lanes that keep their whole
  // row (chunks before the end of a large tie quota, e.g. the zeros of post-ReLU data at a low
  // ratio) all start a multiple of 32 words apart and every store of the gather is a 32-way
  // bank conflict.
  const uint32_t rbase = smem_u32(region);
  auto swz = [](uint32_t addr) -> uint32_t { return addr ^ ((addr >> 5) & 0x7Cu); };
  const bool lined_up = total + mis <= static_cast<uint32_t>(32 * EPR);
  uint32_t pa = rbase + (lane_pre + (lined_up ? mis : 0u)) * static_cast<uint32_t>(sizeof(E));
  auto put = [&](uint32_t v) {
    if (DT == 0) asm volatile("st.shared.u32 [%0], %1;" ::"r"(swz(pa)), "r"(v) : "memory");
    else asm volatile("st.shared.u16 [%0], %1;" ::"r"(swz(pa)), "h"(static_cast<unsigned short>(v)) : "memory");
    pa += static_cast<uint32_t>(sizeof(E));
  };
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint32_t c[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (DT == 0) {
        if ((word[0] >> (4 * j + i)) & 1u) put(c[i]);
      } else {
        const int e = 8 * j + 2 * i;
        if ((word[(e >> 5) % WPL] >> (e & 31)) & 1u) put(c[i]);
        if ((word[(e >> 5) % WPL] >> ((e + 1) & 31)) & 1u) put(c[i] >> 16);
      }
    }
  }
  __syncwarp();
  auto elem_at = [&](uint32_t i) -> E {          // packed element i of the region
    E v;
    const uint32_t addr = swz(rbase + i * static_cast<uint32_t>(sizeof(E)));
    if (DT == 0) { uint32_t u; asm volatile("ld.shared.u32 %0, [%1];" : "=r"(u) : "r"(addr) : "memory"); v = static_cast<E>(u); }
    else { unsigned short u; asm volatile("ld.shared.u16 %0, [%1];" : "=h"(u) : "r"(addr) : "memory"); v = static_cast<E>(u); }
    return v;
  };
  if (lined_up) {
    // slots [mis, mis + total) of the region go to gbase[mis ...]; gbase is 16-byte aligned
    E* gbase = values + (kept_before - mis);
    const uint32_t end = mis + total;
    const uint32_t v_first = mis ? 1u : 0u;    // first whole vector
    const uint32_t v_end = end / EPV;          // one past the last whole vector
    if (mis) {
      const uint32_t sl = mis + lane;
      if (sl < static_cast<uint32_t>(EPV) && sl < end &&
          SURGEON_IN_BOUNDS(kept_before - mis + sl, n_stored, &a.hdr->status))
        gbase[sl] = elem_at(sl);
    }
    for (uint32_t g = v_first + lane; g < v_end; g += 32) {
      // the four words of a vector share their row: one 16-byte load, words permuted by the XOR
      const uint32_t la = rbase + g * 16u;
      const uint32_t xr = (la >> 5) & 0x7Cu;
      uint4 u;
      asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                   : "=r"(u.x), "=r"(u.y), "=r"(u.z), "=r"(u.w) : "r"(la ^ (xr & 0x70u)) : "memory");
      if (xr & 4u) { uint32_t t = u.x; u.x = u.y; u.y = t; t = u.z; u.z = u.w; u.w = t; }
      if (xr & 8u) { uint32_t t = u.x; u.x = u.z; u.z = t; t = u.y; u.y = u.w; u.w = t; }
      if (SURGEON_IN_BOUNDS(kept_before - mis + g * EPV + EPV - 1, n_stored, &a.hdr->status))
        *reinterpret_cast<uint4*>(gbase + g * EPV) = u;
    }
    const uint32_t t0 = (v_end > v_first ? v_end : v_first) * EPV;
    if (t0 + lane < end && SURGEON_IN_BOUNDS(kept_before - mis + t0 + lane, n_stored, &a.hdr->status))
      gbase[t0 + lane] = elem_at(t0 + lane);
  } else {
    // a full chunk with a misaligned destination: no room for the shift, element-wise vectors
    E* dst = values + kept_before;
    uint32_t head = mis ? EPV - mis : 0;
    if (head > total) head = total;
    const uint32_t n_vec = (total - head) / EPV;
    if (lane < head && SURGEON_IN_BOUNDS(kept_before + lane, n_stored, &a.hdr->status))
      dst[lane] = elem_at(lane);
    for (uint32_t v = lane; v < n_vec; v += 32) {
      const uint32_t b = head + v * EPV;
      uint4 o;
      if (DT == 0) {
        o = make_uint4(elem_at(b), elem_at(b + 1), elem_at(b + 2), elem_at(b + 3));
      } else {
        o = make_uint4(elem_at(b) | (static_cast<uint32_t>(elem_at(b + 1)) << 16),
                       elem_at(b + 2) | (static_cast<uint32_t>(elem_at(b + 3)) << 16),
                       elem_at(b + 4) | (static_cast<uint32_t>(elem_at(b + 5)) << 16),
                       elem_at(b + 6) | (static_cast<uint32_t>(elem_at(b + 7)) << 16));
      }
      if (SURGEON_IN_BOUNDS(kept_before + head + v * EPV + EPV - 1, n_stored, &a.hdr->status))
        *reinterpret_cast<uint4*>(dst + head + v * EPV) = o;
    }
    const uint32_t done = head + n_vec * EPV;
    if (lane < total - done && SURGEON_IN_BOUNDS(kept_before + done + lane, n_stored, &a.hdr->status))
      dst[done + lane] = elem_at(done + lane);
  }
  return true;
}

// ---- searching a histogram of kSelBins bins from its top ---------------------------------------------
// Thread t holds bin kSelBins - 1 - t (threads past the bins: 0); returns the count above its bin.
// `total` (every thread): the sum of all bins.  One barrier inside, one due before s_warp is used again.
__device__ __forceinline__ uint32_t count_above_mine(uint32_t b, uint32_t* s_warp, uint32_t* total) {
  const uint32_t excl = warp_excl_scan(b);
  const int warp = threadIdx.x >> 5;
  if (lane_id() == 31) s_warp[warp] = excl + b;
  __syncthreads();
  const uint32_t mine = lane_id() < kWarps ? s_warp[lane_id()] : 0u;
  const uint32_t before = warp_excl_scan(mine);
  *total = __shfl_sync(kFull, before, 31);       // (lanes past the warps add nothing)
  return excl + __shfl_sync(kFull, before, warp);
}
// The bin with #(bins above) < want <= #(bins >= it): its thread stores it, the count above it and its own.
__device__ __forceinline__ void place_rank(uint32_t b, uint32_t above, uint32_t want, uint32_t* res) {
  if (above < want && want <= above + b) {
    res[0] = static_cast<uint32_t>(kSelBins - 1 - static_cast<int>(threadIdx.x));
    res[1] = above;
    res[2] = b;
  }
}
__device__ __forceinline__ uint32_t my_bin(const uint32_t* hist) {
  return threadIdx.x < kSelBins ? hist[kSelBins - 1 - threadIdx.x] : 0u;
}

// The first n_in keys of a slot in shared memory, f(key), a warp together.
template <int DT, typename F>
__device__ __forceinline__ void slot_keys_warp(const typename Elem<DT>::type* slot, uint32_t n_in, F f) {
  for (uint32_t i = lane_id(); i < n_in; i += 32) f(static_cast<uint32_t>(slot[i]));
}
// Of slots in global memory: f(c, acc, key) for the listed keys of chunks 0 .. n_local - 1, then done(c, cnt[c],
// the chunk's acc) on one lane.  Half a warp per chunk, 8 bytes per lane (32 fp32 or 64 bf16 keys; few chunks
// have more) and four chunks in flight: one trip to L2 for 128 chunks.  (A lane per chunk, 64 bytes at a time,
// took 5-7 us a call.)  Of a larger tensor (`many`) a lane per chunk, which has four times as many chunks in
// flight and asks for little more than the keys: 128 at a time made 4.3 GB 6 % slower.
template <int DT, typename F, typename D>
__device__ __forceinline__ void slot_keys_global(const typename Elem<DT>::type* slots, const uint32_t* cnt, int n_local, bool many, F f, D done) {
  if (many) {
    constexpr uint32_t EPV = 16 / sizeof(typename Elem<DT>::type);
    for (int c = threadIdx.x; c < n_local; c += kThreads) {
      const uint32_t v = cnt[c], n_in = min(v >> 16, static_cast<uint32_t>(slot_entries(DT)));
      uint32_t acc = 0;
      const uint4* p = reinterpret_cast<const uint4*>(slots + static_cast<long long>(c) * slot_entries(DT));
      for (uint32_t v0 = 0; v0 * EPV < n_in; v0 += 4) {
        uint4 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = (v0 + u) * EPV < n_in ? p[v0 + u] : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t w[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
#pragma unroll
          for (uint32_t e = 0; e < EPV; ++e)
            if ((v0 + u) * EPV + e < n_in) f(c, acc, (DT == 0) ? w[e % 4] : (w[e >> 1] >> (16 * (e & 1))) & 0xFFFFu);
        }
      }
      done(c, v, acc);
    }
    return;
  }
  constexpr uint32_t EPW = 8 / sizeof(typename Elem<DT>::type);     // keys of a lane
  constexpr int kFlight = 4;
  const uint32_t hl = threadIdx.x & 15u;
  for (int c0 = (threadIdx.x >> 5) * 2; c0 < n_local; c0 += kFlight * (kThreads / 16)) {
    const int cf = c0 + static_cast<int>((threadIdx.x >> 4) & 1u);
    uint32_t v[kFlight];
    uint2 q[kFlight];
#pragma unroll
    for (int u = 0; u < kFlight; ++u) {
      const int c = cf + u * (kThreads / 16);
      v[u] = c < n_local ? cnt[c] : 0u;
      const uint2* p = reinterpret_cast<const uint2*>(slots + static_cast<long long>(c) * slot_entries(DT)) + hl;
      q[u] = hl * EPW < (v[u] >> 16) ? *p : make_uint2(0, 0);
    }
#pragma unroll
    for (int u = 0; u < kFlight; ++u) {
      const int c = cf + u * (kThreads / 16);
      const uint32_t n_in = min(v[u] >> 16, static_cast<uint32_t>(slot_entries(DT)));
      uint32_t acc = 0;
#pragma unroll
      for (uint32_t e = 0; e < EPW; ++e) {
        const uint32_t w = (DT == 0 ? e : e >> 1) ? q[u].y : q[u].x;
        if (hl * EPW + e < n_in) f(c, acc, DT == 0 ? w : (w >> (16 * (e & 1))) & 0xFFFFu);
      }
#pragma unroll 1
      for (uint32_t i = 16 * EPW + hl; i < n_in; i += 16)
        f(c, acc, static_cast<uint32_t>(slots[static_cast<long long>(c) * slot_entries(DT) + i]));
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
      if (hl == 0 && c < n_local) done(c, v[u], acc);
    }
  }
}

// ---- the kernel -----------------------------------------------------------------------------------
// What CTA 0 answers at an exchange: the next bracket, the count of keys above it, and what to do.
enum Step : uint32_t {
  kRead = 0,       // count the bracket in another pass over the chunks
  kRefine = 1,     // count it from the lists
  kKeys = 2,       // few enough listed keys lie inside: report them
  kZero = 3,       // the threshold is 0: whatever is neither above nor inside the last bracket is a tie
  kOneKey = 4,     // the threshold is lo, the only key inside the last bracket: the counts stand
  kListed = 5,     // the threshold is lo; the lists complete the counts
  kRecount = 6,    // the threshold is lo; the lists overflowed: count once more
};

// CTA 0: the answers of a phase and the histogram of a round, before the exchange that leads to them.
__device__ __forceinline__ void prepare_phase(const PruneArgs& a, int phase) {
  if (phase < kSelPhases)
    for (int i = threadIdx.x; i < kSelMaxCtas + 2; i += kThreads) a.answer[phase * (kSelMaxCtas + 2) + i].x = 0ull;
}
__device__ __forceinline__ void prepare_round(const PruneArgs& a, int round) {
  if (round < kSelHists && threadIdx.x < kSelBins) a.hist[round * kSelBins + threadIdx.x] = 0u;
}

// RES: the CTA's whole range stays in the ring (at most kResidentChunks chunks per CTA).
template <int DT, bool RES>
__global__ void __launch_bounds__(kThreads, 1)
prune_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ PruneArgs a) {
  using E = typename Elem<DT>::type;
  constexpr uint32_t kMask = Elem<DT>::kKeyMask;
  constexpr uint32_t kKeyMax = kMask;
  constexpr int EPR = 128 / sizeof(E);
  constexpr int WPL = EPR / 32;
  constexpr int EPV = 16 / sizeof(E);
  constexpr int kSlot = slot_entries(DT);
  static_assert(kSlot * sizeof(E) == kSlotBytes, "slot size");
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* ring = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* aux = ring + kRingBytes;
  uint32_t* hist = reinterpret_cast<uint32_t*>(aux);
  __shared__ __align__(8) unsigned long long bars[kResidentChunks];
  __shared__ uint32_t s_warp[kWarps];
  __shared__ unsigned long long s_warp64[kWarps];
  __shared__ uint32_t s_res[8];
  __shared__ uint32_t s_tot[4];                // keys above / inside the bracket, largest key inside, largest ~key inside
  __shared__ uint32_t s_over, s_fail, s_nkeys;
  __shared__ unsigned long long s_ans[2];
  __shared__ uint32_t s_bin_key[kMaxKeys];      // the keys that this CTA reports at the last exchange,
  __shared__ int s_bin_chunk[kMaxKeys];        // and their chunks

  const int tid = threadIdx.x;
  const int warp = tid >> 5;
  const uint32_t lane = lane_id();
  const int G = static_cast<int>(gridDim.x);
  const bool master = blockIdx.x == 0;
  const int c_begin = static_cast<int>(static_cast<long long>(a.n_chunks) * blockIdx.x / G);
  const int c_end = static_cast<int>(static_cast<long long>(a.n_chunks) * (blockIdx.x + 1) / G);
  const int n_local = c_end - c_begin;
  // Of a gigabyte tensor (a.spread) the warps claim their chunks four at a time, in either pass: equal
  // shares took some SMs 620 us and others 760, and all wait for the last.  Four sets of CTAs claim
  // from counters of their own (one counter for all passes on a claim every 3 ns, too slow).  Only
  // what is counted and placed per CTA stays a contiguous range then.
  const bool spread = !RES && a.spread != 0;
  const int n_mine = warp < n_local ? (n_local - 1 - warp) / kWarps + 1 : 0;   // (not spread) chunks c_begin + warp + 16 i
  uint32_t* cnt = spread ? a.cnt + c_begin : reinterpret_cast<uint32_t*>(aux + kAuxCnt);
  unsigned long long* prefix =
      spread ? a.prefix + c_begin : reinterpret_cast<unsigned long long*>(aux + kAuxPrefix);
  E* s_slots = reinterpret_cast<E*>(aux + kAuxSlots);     // RES: the chunks' slots, else a staging slot per warp
  E* g_slots = reinterpret_cast<E*>(a.slots) + static_cast<long long>(c_begin) * kSlot;
  const E* __restrict__ x = reinterpret_cast<const E*>(a.x);

  // ---- the ring: this warp's places ----
  unsigned char* my_ring = ring + warp * (kSlotsPerWarp * kChunkBytes);
  const uint32_t my_bars = smem_u32(bars + warp * kSlotsPerWarp);
  uint32_t parity = 0;                           // bit s: phase of place s's next wait
  auto chunk_of = [&](int i) { return c_begin + warp + kWarps * i; };
  auto issue = [&](int c, int s) {               // start the load of chunk c into place s (one lane)
    if (lane == 0 && static_cast<long long>(c) * 32 < a.n_rows_full) {
      tc::mbar_arrive_expect_tx(my_bars + 8 * s, kChunkBytes);
      tc::tma_load_2d(smem_u32(my_ring + s * kChunkBytes), &xmap, 0, c * 32, my_bars + 8 * s);
    }
  };
  auto arrived = [&](int c, int s) -> bool {     // wait for it; the tensor's last, partial row is added
    unsigned char* region = my_ring + s * kChunkBytes;
    const long long row0 = static_cast<long long>(c) * 32;
    if (row0 < a.n_rows_full) {
      if (!tc::mbar_wait(my_bars + 8 * s, (parity >> s) & 1u)) return false;
      parity ^= 1u << s;
    } else {
      for (int v = lane; v < kChunkBytes / 16; v += 32)
        *reinterpret_cast<uint4*>(region + v * 16) = make_uint4(0, 0, 0, 0);
      tc::fence_proxy_async();                   // (these stores precede the next TMA fill of the place)
      __syncwarp();
    }
    if (row0 + 32 > a.n_rows_full && a.n > a.n_rows_full * EPR) {
      const int r = static_cast<int>(a.n_rows_full - row0);       // the map fills the rows past it with zeros
      for (int e = lane; e < static_cast<int>(a.n - a.n_rows_full * EPR); e += 32) {
        const int byte = e * static_cast<int>(sizeof(E));
        *reinterpret_cast<E*>(region + r * 128 + (((byte >> 4) ^ (r & 7)) << 4) + (byte & 15)) =
            x[a.n_rows_full * EPR + e];
      }
      tc::fence_proxy_async();
      __syncwarp();
    }
    return true;
  };
  // The warp's chunks of one pass in the order of their loads: next() is the next one, or n_chunks.
  static_assert(kSlotsPerWarp == 3, "three loads in flight");
  int fly0 = a.n_chunks, fly1 = a.n_chunks, fly2 = a.n_chunks;    // chunks in flight, the oldest first
  int at_i = 0, claim = 0, pass = 0;             // (not spread) index of the next one; (spread) the claimed group; passes begun
  uint32_t ahead = 0;                            // (lane 0) the group claimed one chunk ahead
  auto next = [&]() -> int {
    if (!spread) return at_i < n_mine ? chunk_of(at_i++) : a.n_chunks;
    if ((at_i & 3) == 0) {
      // the first group of a pass is the warp's own, the others are claimed
      const int n_sets = min(kClaimSets, G), set = static_cast<int>(blockIdx.x) * n_sets / G;
      const int set_begin = (set * G + n_sets - 1) / n_sets, set_end = ((set + 1) * G + n_sets - 1) / n_sets;
      uint32_t g = (blockIdx.x - set_begin) * kWarps + warp;
      if (at_i > 0) g = (set_end - set_begin) * kWarps + __shfl_sync(kFull, ahead, 0);
      claim = static_cast<int>(min(4u * (g * n_sets + set), static_cast<uint32_t>(a.n_chunks)));
    }
    if ((at_i & 3) == 3 && lane == 0) {          // the round trip hides behind a chunk
      const int set = static_cast<int>(blockIdx.x) * min(kClaimSets, G) / G;
      ahead = atomicAdd(&a.claims[(pass * kClaimSets + set) * kClaimStride], 1u);
    }
    const int c = claim + (at_i++ & 3);
    return c < a.n_chunks ? c : a.n_chunks;
  };
  auto begin_pass = [&](bool reverse) {          // the first three loads; reverse: from the tensor's end
    at_i = 0;
    auto one = [&](int s) -> int {
      int c = next();
      if (c < a.n_chunks) {
        if (reverse) c = a.n_chunks - 1 - c;
        issue(c, s);
      }
      return c;
    };
    fly0 = one(0); fly1 = one(1); fly2 = one(2);
  };
  // A wait gave up: the loads behind it are waited for (with a limit) as well.
  auto give_up = [&](int s) {
    s_fail = 1;
    if (fly1 < a.n_chunks) arrived(fly1, (s + 1) % 3);
    if (fly2 < a.n_chunks) arrived(fly2, (s + 2) % 3);
  };
  // One pass over the warp's chunks: f(chunk, region) is true where it wrote to the region.
  auto run_pass = [&](bool reverse, auto f) {
    for (int s = 0; fly0 < a.n_chunks; s = s == 2 ? 0 : s + 1) {
      unsigned char* region = my_ring + s * kChunkBytes;
      if (!arrived(fly0, s)) { give_up(s); break; }
      const bool written = f(fly0, region);
      fly0 = fly1; fly1 = fly2;
      int c = next();
      if (c < a.n_chunks) {
        if (reverse) c = a.n_chunks - 1 - c;
        if (written) tc::fence_proxy_async();    // this warp's writes to the place precede the next TMA fill
        __syncwarp();                            // every lane has read the place
        issue(c, s);
      }
      fly2 = c;
    }
    ++pass;
  };
  // (RES) the chunks are where the first loads put them.
  auto run_resident = [&](bool loading, auto f) {
    for (int i = 0; i < n_mine; ++i) {
      if (loading && !arrived(chunk_of(i), i)) { s_fail = 1; for (++i; i < n_mine; ++i) arrived(chunk_of(i), i); break; }
      f(chunk_of(i), my_ring + i * kChunkBytes);
    }
  };
  auto drain = [&]() {                           // before leaving with the first loads under way
    if (fly0 < a.n_chunks) arrived(fly0, 0);
    if (fly1 < a.n_chunks) arrived(fly1, 1);
    if (fly2 < a.n_chunks) arrived(fly2, 2);
  };
  int phase = 1;                                 // of the next exchange
  auto meet = [&]() -> bool {                    // an exchange without a message: what was written before is visible after
    __syncthreads();
    if (tid == 0) {
      fence_gpu();
      word_store(a.arrive + phase * kSelMaxCtas + blockIdx.x, a.token, 0ull);
    }
    int ok = 1;
    unsigned long long ignored;
    if (master) {
      if (tid < G) {
        ok = word_wait(a.arrive + phase * kSelMaxCtas + tid, a.token, &ignored);
        fence_gpu();
        a.arrive[phase * kSelMaxCtas + tid].x = 0ull;
      }
      prepare_phase(a, phase + 1);
      ok = __syncthreads_and(ok);
      if (ok && tid == 0) {
        fence_gpu();
        word_store(a.answer + phase * (kSelMaxCtas + 2), a.token, 0ull);
      }
    } else {
      if (tid == 0) {
        ok = word_wait(a.answer + phase * (kSelMaxCtas + 2), a.token, &ignored);
        fence_gpu();
      }
      ok = __syncthreads_and(ok);
    }
    ++phase;
    return ok != 0;
  };
  // The whole CTA leaves after a wait gave up.  It takes back what it has stored for the others: a replay of a
  // captured call carries the same token and must not find it.
  auto quit = [&]() {
    if (tid == 0) atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
    if (tid < kSelPhases) a.arrive[tid * kSelMaxCtas + blockIdx.x].x = 0ull;
    if (master)
      for (int i = tid; i < kSelPhases * (kSelMaxCtas + 2); i += kThreads) a.answer[i].x = 0ull;
  };

  // ---- set-up ----
  if (lane == 0) {                               // a warp's barriers are its own
    for (int s = 0; s < kSlotsPerWarp; ++s) tc::mbar_init(my_bars + 8 * s, 1);
    tc::fence_barrier_init();
  }
  __syncwarp();
  begin_pass(false);
  if (tid == 0) {
    s_fail = 0;
    s_over = 0;
  }
  if (tid < 4) s_tot[tid] = 0;
  for (int i = tid; i < kSampleBytes / 16; i += kThreads) reinterpret_cast<uint4*>(aux)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();

  // ---- the sample ----
  // A resident tensor: 2048 vectors of 32 (fp32) or 16 (bf16) bytes, one per stratum, the same for
  // every CTA (each starts elsewhere in it, so that they do not all ask for the same lines at the
  // same time).  More would not pay: 148 CTAs that read 8192 places took 12 us.  The margin is 4
  // standard deviations (a miss costs a round).
  // A larger tensor, for which a miss is another read of it and a narrow bracket pays: every CTA
  // samples the whole tensor at places of its own (stratum G i + p of the G i-th row, p scrambled from
  // row to row so that no period of the data falls to one CTA) and reports where the threshold lies in
  // its own 4 or 8 thousand elements.  The CTAs' answers are independent draws whose median is the
  // threshold, however the elements are distributed, so the ones 2.5 sqrt(G) places (5 standard
  // deviations) to either side of the middle bound it: 0.4 % of the elements to each side, as the sum of
  // all histograms would give.  One exchange of one word per CTA, 4 us less than a window from CTA 0's part
  // and added-up histograms took.
  uint32_t lo = 1, hi = kKeyMax;
  const uint32_t n_vec = static_cast<uint32_t>(a.n / EPV);
  constexpr int kPer = RES ? (DT == 0 ? 8 : 4) : 2;       // vectors per thread
  constexpr int kBinShift = Elem<DT>::kKeyBits - kSampleBinsLog2;
  constexpr int kFineShift = kBinShift > kSelBinsLog2 ? kBinShift - kSelBinsLog2 : 0;     // (!RES)
  uint4 v[kPer];
  {
    constexpr uint32_t kStrata = kPer * kThreads / (DT == 0 ? 2 : 1);     // of this CTA
    const uint32_t strata = RES ? kStrata : kStrata * G;
    const float stride = static_cast<float>(n_vec) / static_cast<float>(strata);
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      uint32_t loc = u * kThreads + tid, part = 0;
      if (DT == 0) { part = loc & 1u; loc >>= 1; }         // two lanes share a stratum: 32 bytes
      if (RES) {
        loc = (loc + blockIdx.x * 37u) % kStrata;
      } else {
        const uint32_t at_row = blockIdx.x + __umulhi(hash_u32(loc + 0x9E3779B9u), static_cast<uint32_t>(G));
        loc = loc * G + (at_row >= static_cast<uint32_t>(G) ? at_row - G : at_row);
      }
      const float at = (static_cast<float>(loc) + static_cast<float>(hash_u32(loc) >> 8) * (1.0f / 16777216.0f)) * stride;
      uint32_t pos = static_cast<uint32_t>(at);
      if (DT == 0) pos = (pos & ~1u) + part;
      v[u] = n_vec ? __ldg(reinterpret_cast<const uint4*>(a.x) + min(pos, n_vec - 1)) : make_uint4(0, 0, 0, 0);
    }
  }
  if (master) {                                  // meanwhile CTA 0 prepares the exchange
    if (tid == 0) {                              // (no value yet: what reads the store trusts the count)
      a.hdr->status = SURGEON_OK;
      a.hdr->n_keep = 0;
    }
    prepare_phase(a, 1);
    prepare_round(a, 0);
    if (!RES && tid < kSelPhases * kClaimSets) a.claims[tid * kClaimStride] = 0u;
    if (RES) {
      __syncthreads();
      if (tid == 0) {
        fence_gpu();
        word_store(a.answer, a.token, 0ull);     // phase 0: the histogram is zero, the header begun
      }
    }
  }
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
    for (int e = 0; e < EPV; ++e) {
      const uint32_t key = ((DT == 0) ? w[e % 4] : (w[e >> 1] >> (16 * (e & 1)))) & kMask;
      const uint32_t bin = key >> kBinShift;
      if (key) atomicAdd(&hist[bin >> 1], 1u << (16 * (bin & 1)));   // (not the zeros, half of post-ReLU data)
    }
  }
  // rank of the threshold inside the sample, and (RES) a margin of some standard deviations of a binomial count
  const float q = static_cast<float>(a.k) / static_cast<float>(a.n);
  constexpr float kOwn = static_cast<float>(kPer * kThreads * EPV);        // elements in this CTA's histogram
  const float up = q * kOwn, down = kOwn - up;   // of them above and below the threshold
  const bool no_hi = up < 16.0f, no_lo = down < 16.0f;     // (!RES) too few for a median that means something:
  uint32_t r_hi, r_lo = 0;                       // that side stays open, and the rank moves to the other
  if (RES) {
    const float delta = 4.0f * sqrtf(kOwn * q * (1.0f - q)) + 16.0f;
    r_hi = up - delta >= 1.0f ? static_cast<uint32_t>(up - delta) : 0u;                        // 0: none
    r_lo = up + delta <= kOwn - 1.0f ? static_cast<uint32_t>(up + delta) + 1u : 0u;            // 0: none
  } else {
    r_hi = static_cast<uint32_t>(no_hi ? up + sqrtf(up) + 2.0f : no_lo ? up - sqrtf(down) - 2.0f : up + 0.5f);
  }
  if (tid < 2) s_res[tid] = RES && tid == 0 && r_hi == 0 ? kSampleBins - 1u : 0u;
  __syncthreads();
  {
    // the bins of the ranks in the CTA's own histogram
    // thread t owns the 32 bins below 2^14 - 32 t
    const uint4* mine = reinterpret_cast<const uint4*>(hist) + 4 * (kSampleBins / 32 - 1 - tid);
    uint32_t sum = 0;
    if (tid < kSampleBins / 32) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {              // (started at a lane-dependent vector: no bank conflicts)
        const uint4 h = mine[(j + (lane >> 1)) & 3];
        sum += (h.x & 0xFFFFu) + (h.x >> 16) + (h.y & 0xFFFFu) + (h.y >> 16) + (h.z & 0xFFFFu) + (h.z >> 16) +
               (h.w & 0xFFFFu) + (h.w >> 16);
      }
    }
    uint32_t all;
    const uint32_t above = count_above_mine(sum, s_warp, &all);
#pragma unroll 1
    for (int which = 0; which < (RES ? 2 : 1); ++which) {
      // (a rank among the zeros lies below every counted bin: bin 0)
      const uint32_t want = which ? r_lo : r_hi;
      if (want && above < want && want <= above + sum) {
        uint32_t acc = above;
        int bin = 31;
#pragma unroll 1
        for (; bin > 0; --bin) {
          const uint32_t c = (reinterpret_cast<const uint32_t*>(mine)[bin >> 1] >> (16 * (bin & 1))) & 0xFFFFu;
          if (acc + c >= want) break;
          acc += c;
        }
        s_res[which] = static_cast<uint32_t>(kSampleBins - 32 - 32 * tid + bin);
        if (!RES) s_res[1] = want - acc;         // the rank among the bin's elements
      }
    }
    __syncthreads();
  }
  if (RES) {
    lo = max(s_res[1] << kBinShift, 1u);
    hi = (s_res[0] << kBinShift) | ((1u << kBinShift) - 1u);
  } else {
    // the key's next bits, among the bin's elements (a bin holds about as many elements as the bracket will)
    const uint32_t bin = s_res[0], want = s_res[1];
    if (tid < kSelBins) hist[tid] = 0;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
      for (int e = 0; e < EPV; ++e) {
        const uint32_t key = ((DT == 0) ? w[e % 4] : (w[e >> 1] >> (16 * (e & 1)))) & kMask;
        if (key && key >> kBinShift == bin) atomicAdd(&hist[(key & ((1u << kBinShift) - 1u)) >> kFineShift], 1u);
      }
    }
    if (tid == 0) s_res[3] = 0;
    __syncthreads();
    uint32_t all;
    const uint32_t b = my_bin(hist);
    const uint32_t above = count_above_mine(b, s_warp, &all);
    if (want) place_rank(b, above, want, s_res + 3);
    __syncthreads();
    if (tid == 0)                                // phase 0: where it lies
      word_store(a.arrive + blockIdx.x, a.token, want ? (bin << (kBinShift - kFineShift)) | s_res[3] : 0u);
    unsigned long long w = 0;
    int ok = 1;
    if (master) {
      uint32_t* bins = hist;                     // (the sample is done with)
      if (tid < G) {
        ok = word_wait(a.arrive + tid, a.token, &w);
        a.arrive[tid].x = 0ull;
      }
      // distinct, in the keys' order
      if (tid < kSelMaxCtas) bins[tid] = tid < G ? (static_cast<uint32_t>(w) << 8) | (kSelMaxCtas - 1u - tid) : 0u;
      if (!__syncthreads_and(ok)) { drain(); quit(); return; }
      const int margin = static_cast<int>(2.5f * sqrtf(static_cast<float>(G))) + 1;
      const int at_hi = G / 2 - margin, at_lo = G / 2 + margin;
      if (tid < G) {
        const uint32_t my = bins[tid];
        int larger = 0;
#pragma unroll 4
        for (int i = 0; i < (G + 3) / 4; ++i) {
          const uint4 o = reinterpret_cast<const uint4*>(bins)[i];
          larger += (o.x > my ? 1 : 0) + (o.y > my ? 1 : 0) + (o.z > my ? 1 : 0) + (o.w > my ? 1 : 0);
        }
        if (larger == at_hi) s_res[0] = my >> 8;
        if (larger == at_lo) s_res[1] = my >> 8;
      }
      __syncthreads();
      hi = no_hi || at_hi < 0 ? kKeyMax : (s_res[0] << kFineShift) | ((1u << kFineShift) - 1u);
      lo = no_lo || at_lo >= G ? 1u : max(s_res[1] << kFineShift, 1u);
      if (tid == 0) {
        fence_gpu();                             // the histogram is zero, the claims, the header begun
        word_store(a.answer, a.token, lo | (static_cast<unsigned long long>(hi) << 32));
      }
    } else {
      if (tid == 0) {
        ok = word_wait(a.answer, a.token, &w);
        fence_gpu();
        s_ans[0] = w;
      }
      if (!__syncthreads_and(ok)) { drain(); quit(); return; }
      lo = static_cast<uint32_t>(s_ans[0]);
      hi = static_cast<uint32_t>(s_ans[0] >> 32);
    }
  }

  // ---- the threshold ----
  // Every round counts the keys of [lo, hi] in bins of 2^shift keys, either in a pass over the chunks
  // (kRead) or from the keys that the last such pass listed (kRefine).
  uint32_t step = kRead, n_above = 0;            // n_above: keys above hi
  bool listed = false, loaded = true;            // (CTA 0) the last pass's lists are complete
  int shift = 0;
  int round = 0;
  uint32_t tau = 0, n_greater = 0;
  unsigned long long before = 0;
  for (;;) {
  for (; step <= kRefine; ++round) {
    const uint32_t range = hi - lo;
    shift = max(0, 32 - __clz(range) - kSelBinsLog2);
    __syncthreads();
    if (tid < kSelBins) hist[tid] = 0;
    if (step == kRead) {
      if (tid < 4) s_tot[tid] = 0;
      if (tid == 0) s_over = 0;
    }
    __syncthreads();
    if (step == kRead) {
      if (!RES && !loaded) {                     // the pass starts over
        tc::fence_proxy_async();
        __syncwarp();
        begin_pass(false);
      }
      uint32_t w_above = 0;
      uint32_t kmax = 0, kinv = 0;               // largest key inside the bracket seen by this lane, and largest ~key
      const uint32_t c_above = ge_const(hi + 1u), c_lo = ge_const(lo);
      auto classify = [&](int c, unsigned char* region) -> bool {
        const int cl = c - c_begin;              // the chunk's place in the CTA's range (spread: anywhere)
        uint4 q[8];
        load_row(region, q);
        // (rows and elements past the tensor's end hold key 0: below every bracket)
        uint32_t cw[WPL], ac = 0, cc = 0;
        if (DT == 0) {
          // the sign bit of (hi - key) says key > hi, that of (key - lo) says key < lo (see mask_ge)
          uint32_t aw = 0, lw = 0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t w[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const uint32_t key = w[e] & kMask;
              aw = __funnelshift_l(hi - key, aw, 1);
              lw = __funnelshift_l(key - lo, lw, 1);
            }
          }
          ac = __popc(aw);
          cw[0] = __brev(~lw & ~aw);
        } else {
          uint32_t ga[WPL], gl[WPL];
#pragma unroll
          for (int w = 0; w < WPL; ++w) { ga[w] = 0; gl[w] = 0; }
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t w[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int pw = 4 * j + e;           // packed word of the row: elements 2pw, 2pw + 1
              const uint32_t keys2 = w[e] & 0x7FFF7FFFu;
              ga[(pw >> 4) % WPL] |= pair_flags(keys2, c_above, pw & 15);
              gl[(pw >> 4) % WPL] |= pair_flags(keys2, c_lo, pw & 15);
            }
          }
#pragma unroll
          for (int w = 0; w < WPL; ++w) {
            ac += __popc(ga[w]);
            const uint32_t in = gl[w] & ~ga[w];
            cw[w] = in ? pairs_to_element_order(in) : 0u;
          }
        }
#pragma unroll
        for (int w = 0; w < WPL; ++w) cc += __popc(cw[w]);
        const uint32_t both = __reduce_add_sync(kFull, ac | (cc << 16));   // a chunk has at most 2048 elements
        const uint32_t a_tot = both & 0xFFFFu, c_tot = both >> 16;
        if (lane == 0) cnt[cl] = both;
        w_above += a_tot;
        if (c_tot > static_cast<uint32_t>(kSlot)) {
          // Massive ties.  If the chunk's keys inside the bracket all are one key, it is counted in
          // one go; if that holds everywhere with the same key, it is the threshold and the counts
          // are final without a list.
          const uint32_t k1 = one_key_of_chunk<DT>(region, cw[0], cw[WPL - 1], c_tot);
          if (lane == 0) s_over = 1;
          if (k1) {
            if (lane == 0) atomicAdd(&hist[(k1 - lo) >> shift], c_tot);
            kmax = max(kmax, k1);
            kinv = max(kinv, ~k1);
          } else {
#pragma unroll
            for (int w = 0; w < WPL; ++w) {
              for (uint32_t m = cw[w]; m; m &= m - 1) {
                const uint32_t key = row_elem<DT>(region, 32 * w + __ffs(m) - 1) & kMask;
                atomicAdd(&hist[(key - lo) >> shift], 1u);
              }
            }
            kmax = kinv = 0xFFFFFFFFu;
          }
        } else if (c_tot) {
          // the lanes put their keys into the slot, then share the rest of the work evenly
          E* sl = s_slots + (RES ? cl : warp) * kSlot;
          uint32_t pos = warp_excl_scan(cc);
#pragma unroll
          for (int w = 0; w < WPL; ++w)
            for (uint32_t m = cw[w]; m; m &= m - 1)
              sl[pos++] = static_cast<E>(row_elem<DT>(region, 32 * w + __ffs(m) - 1) & kMask);
          __syncwarp();
          for (uint32_t t = lane; t < c_tot; t += 32) {
            const uint32_t key = sl[t];
            atomicAdd(&hist[(key - lo) >> shift], 1u);
            kmax = max(kmax, key);
            kinv = max(kinv, ~key);
            if (!RES) g_slots[static_cast<long long>(cl) * kSlot + t] = static_cast<E>(key);
          }
          __syncwarp();
        }
        return false;
      };
      if (RES) run_resident(loaded, classify);
      else run_pass(false, classify);
      loaded = false;
      kmax = __reduce_max_sync(kFull, kmax);
      kinv = __reduce_max_sync(kFull, kinv);
      if (lane == 0) {
        if (w_above) atomicAdd(&s_tot[0], w_above);
        if (kmax) atomicMax(&s_tot[2], kmax);
        if (kinv) atomicMax(&s_tot[3], kinv);
      }
    } else {
      auto add = [&](uint32_t key) {
        const uint32_t rel = key - lo;           // (below lo: wraps far above the range)
        if (rel <= range) atomicAdd(&hist[rel >> shift], 1u);
      };
      if (RES) {
        for (int c = warp; c < n_local; c += kWarps) slot_keys_warp<DT>(s_slots + c * kSlot, cnt[c] >> 16, add);
      } else {
        slot_keys_global<DT>(g_slots, cnt, n_local, n_local > kThreads / 2, [&](int, uint32_t&, uint32_t key) { add(key); }, [](int, uint32_t, uint32_t) {});
      }
    }
    if (RES && round == 0 && tid == 0) {         // CTA 0 has zeroed the histograms
      unsigned long long ignored;
      if (!word_wait(a.answer, a.token, &ignored)) s_fail = 1;
      fence_gpu();
    }
    __syncthreads();
    if (s_fail) { quit(); return; }
    uint32_t* gh = a.hist + round * kSelBins;
    if (tid < kSelBins) {
      const uint32_t h = hist[tid];
      if (h) atomicAdd(&gh[tid], h);
    }
    __syncthreads();
    if (tid == 0) {
      // reported: keys above, whether a list overflowed, and the one key inside (0: none, ~0: several)
      fence_gpu();
      const uint32_t one = s_tot[2] == 0u ? 0u : (s_tot[2] == ~s_tot[3] ? s_tot[2] : 0xFFFFFFFFu);
      word_store(a.arrive + phase * kSelMaxCtas + blockIdx.x, a.token,
                 (static_cast<unsigned long long>(one) << 32) | s_tot[0] | (s_over << 31));
    }
    if (master) {
      unsigned long long v = 0;
      int ok = 1;
      if (tid < G) {
        ok = word_wait(a.arrive + phase * kSelMaxCtas + tid, a.token, &v, a.stall != 0);
        fence_gpu();                             // (before the clearing: a fence waits for the stores before it)
        a.arrive[phase * kSelMaxCtas + tid].x = 0ull;
      }
      prepare_phase(a, phase + 1);
      prepare_round(a, round + 1);
      if (!__syncthreads_and(ok)) { quit(); return; }
      const uint32_t b = tid < kSelBins ? __ldcg(gh + kSelBins - 1 - tid) : 0u;
      const uint32_t one = static_cast<uint32_t>(v >> 32);
      const uint32_t w_max = __reduce_max_sync(kFull, one), w_inv = __reduce_max_sync(kFull, one ? ~one : 0u);
      const uint32_t w_over = __any_sync(kFull, (static_cast<uint32_t>(v) >> 31) != 0u) ? 1u : 0u;
      const uint32_t w_sum = __reduce_add_sync(kFull, static_cast<uint32_t>(v) & 0x7FFFFFFFu);
      __shared__ uint4 s_red[kWarps];
      if (lane == 0) s_red[warp] = make_uint4(w_sum, w_max, w_inv, w_over);
      uint32_t n_in;
      const uint32_t above = count_above_mine(b, s_warp, &n_in);
      uint32_t sum = 0, key_max = 0, key_inv = 0, over = 0;
      const uint4 red = lane < kWarps ? s_red[lane] : make_uint4(0, 0, 0, 0);
      sum = __reduce_add_sync(kFull, red.x);
      key_max = __reduce_max_sync(kFull, red.y);
      key_inv = __reduce_max_sync(kFull, red.z);
      over = __any_sync(kFull, red.w != 0u) ? 1u : 0u;
      const bool was_read = step == kRead;
      if (was_read) { n_above = sum; listed = over == 0; }
      const long long r = static_cast<long long>(a.k) - n_above;     // rank among the keys of [0, hi]
      if (r < 1) {                               // the bracket lies too low: the threshold is above it
        lo = hi + 1u; hi = kKeyMax; step = kRead;
      } else if (r > n_in) {
        if (lo == 1u) { step = kZero; n_above += n_in; lo = hi = 0; }   // neither above nor inside: zeros
        else { hi = lo - 1u; lo = 1u; step = kRead; }                   // the bracket lies too high
      } else if (was_read && key_max != 0xFFFFFFFFu && key_max == ~key_inv) {
        step = kOneKey; lo = hi = key_max;
      } else {
        place_rank(b, above, static_cast<uint32_t>(r), s_res);
        __syncthreads();
        n_above += s_res[1];
        lo += s_res[0] << shift;
        hi = min(hi, lo + ((1u << shift) - 1u));
        if (shift == 0) step = listed ? kListed : kRecount;
        else if (!listed) step = kRead;
        else step = s_res[2] <= static_cast<uint32_t>(kKeysAtOnce / 2) && shift <= 2 * kSelBinsLog2 ? kKeys : kRefine;
      }
      __syncthreads();
      if (tid == 0) {
        fence_gpu();                             // the cleared words and bins of what comes next
        word_store(a.answer + phase * (kSelMaxCtas + 2), a.token, lo | (static_cast<unsigned long long>(hi) << 32));
        word_store(a.answer + phase * (kSelMaxCtas + 2) + 1, a.token, n_above | (static_cast<unsigned long long>(step) << 32));
        if (phase == 1) a.answer[0].x = 0ull;
      }
    } else {
      if (tid < 2) {
        unsigned long long v = 0;
        if (!word_wait(a.answer + phase * (kSelMaxCtas + 2) + tid, a.token, &v, a.stall != 0)) s_fail = 1;
        if (!RES) fence_gpu();                   // (spread: the counts and lists of the other CTAs)
        s_ans[tid] = v;
      }
      __syncthreads();
      if (s_fail) { quit(); return; }
      lo = static_cast<uint32_t>(s_ans[0]);
      hi = static_cast<uint32_t>(s_ans[0] >> 32);
      n_above = static_cast<uint32_t>(s_ans[1]);
      step = static_cast<uint32_t>(s_ans[1] >> 32);
    }
    ++phase;
    if (round + 1 >= kSelHists && step <= kRefine) {   // cannot happen: a miss, three levels and a pass for ties are the most
      if (tid == 0) atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_INTERNAL));
      return;
    }
  }

  // ---- what this CTA has above the threshold (or above its bin) and at it ----
  if (step == kRecount) {                        // the lists overflowed: count once more from the chunks
    __syncthreads();
    auto recount = [&](int c, unsigned char* region) -> bool {
      uint4 q[8];
      load_row(region, q);
      uint32_t ge[WPL], gt[WPL], g = 0, e = 0;   // (lo >= 1: what lies past the tensor's end is below it)
      mask_ge<DT, WPL>(q, EPR, lo, ge);
      mask_ge<DT, WPL>(q, EPR, lo + 1u, gt);
#pragma unroll
      for (int w = 0; w < WPL; ++w) { g += __popc(gt[w]); e += __popc(ge[w] & ~gt[w]); }
      const uint32_t both = __reduce_add_sync(kFull, g | (e << 16));
      if (lane == 0) cnt[c - c_begin] = both;
      return false;
    };
    if (RES) {
      run_resident(false, recount);
    } else {
      tc::fence_proxy_async();
      __syncwarp();
      begin_pass(false);
      run_pass(false, recount);
    }
    if (spread && !meet()) { quit(); return; }
  }
  if (tid == 0) s_nkeys = 0;
  __syncthreads();
  if (s_fail) { quit(); return; }
  uint32_t n_gt = 0, n_eq = 0;
  if (step == kListed || step == kKeys) {
    // acc: keys above hi, and (upper half) keys of [lo, hi]
    auto report = [&](int c, uint32_t& acc, uint32_t key) {
      if (key > hi) ++acc;
      else if (key >= lo) {
        acc += 0x10000u;
        if (step == kKeys) {
          const uint32_t at = atomicAdd(&s_nkeys, 1u);
          if (at < static_cast<uint32_t>(kMaxKeys)) {
            a.keys[blockIdx.x * kMaxKeys + at] = key;
            s_bin_key[at] = key;
            s_bin_chunk[at] = c;
          }
        }
      }
    };
    auto done = [&](int c, uint32_t v, uint32_t acc) {       // (one lane)
      acc += v & 0xFFFFu;
      if (step == kListed) cnt[c] = acc;
      else prefix[c] = acc & 0xFFFFu;            // (cnt stands: there may be another round)
      n_gt += acc & 0xFFFFu;
      n_eq += acc >> 16;
    };
    if (RES) {
      for (int c = warp; c < n_local; c += kWarps) {
        const uint32_t v = cnt[c];
        uint32_t acc = 0;
        slot_keys_warp<DT>(s_slots + c * kSlot, v >> 16, [&](uint32_t key) { report(c, acc, key); });
        acc = __reduce_add_sync(kFull, acc);
        if (lane == 0) done(c, v, acc);
      }
    } else {
      slot_keys_global<DT>(g_slots, cnt, n_local, n_local > kThreads / 2, report, done);
    }
  } else {
    for (int c = tid; c < n_local; c += kThreads) {
      const uint32_t v = cnt[c];
      uint32_t g = v & 0xFFFFu, e = v >> 16;
      if (step == kZero) {
        const long long left = a.n - static_cast<long long>(c_begin + c) * (32 * EPR);
        g += e;
        e = static_cast<uint32_t>(left < 32 * EPR ? left : 32 * EPR) - g;
        cnt[c] = g | (e << 16);
      }
      n_gt += g;
      n_eq += e;
    }
  }
  n_gt = warp_sum(n_gt);
  n_eq = warp_sum(n_eq);
  if (lane == 0) s_warp64[warp] = (static_cast<unsigned long long>(n_gt) << 32) | n_eq;
  __syncthreads();
  if (tid == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < kWarps; ++w) t += s_warp64[w];
    fence_gpu();
    word_store(a.arrive + phase * kSelMaxCtas + blockIdx.x, a.token, t);
  }

  // ---- last exchange: the threshold, and every CTA's place ----
  tau = lo; n_greater = n_above;
  bool again = false;                            // a CTA has more keys than it can report: narrow the bin first
  if (master) {
    unsigned long long v = 0;
    int ok = 1;
    if (tid < G) {
      ok = word_wait(a.arrive + phase * kSelMaxCtas + tid, a.token, &v);
      fence_gpu();
      a.arrive[phase * kSelMaxCtas + tid].x = 0ull;
    }
    prepare_phase(a, phase + 1);
    if (step == kKeys && tid < kSelBins) hist[tid] = hist[kSelBins + tid] = 0;
    if (!__syncthreads_and(ok)) { quit(); return; }
    if (step == kKeys) {
      const uint32_t n_k = tid < G ? static_cast<uint32_t>(v) : 0u;
      uint32_t* nk = hist + 2 * kSelBins;        // [3][kSelMaxCtas]: keys, above, ties per CTA
      if (tid < kSelMaxCtas) { nk[tid] = n_k; nk[kSelMaxCtas + tid] = 0; nk[2 * kSelMaxCtas + tid] = 0; }
      const uint32_t w_most = __reduce_max_sync(kFull, n_k);
      if (lane == 0) s_warp[warp] = w_most;
      __syncthreads();
      const int most = static_cast<int>(__reduce_max_sync(kFull, lane < kWarps ? s_warp[lane] : 0u));
      __syncthreads();
      constexpr int kPer = kKeysPerThread;
      again = most > kMaxKeys || most * G > kKeysAtOnce;
      if (!again) {
        // (idx / most by multiplication: idx * most < 2^32)
        const uint32_t inv = most > 1 ? 0xFFFFFFFFu / static_cast<uint32_t>(most) + 1u : 0u;
        uint32_t key[kPer];
        int who[kPer];
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
          const int idx = u * kThreads + tid;
          who[u] = most > 1 ? static_cast<int>(__umulhi(static_cast<uint32_t>(idx), inv)) : idx;
          const int i = idx - who[u] * most;
          const bool have = who[u] < G && i < static_cast<int>(nk[min(who[u], kSelMaxCtas - 1)]);
          key[u] = have ? __ldcg(a.keys + who[u] * kMaxKeys + i) : 0u;
        }
        // the rank among them: by the upper bits of key - lo, then by the rest
        const int coarse = shift > kSelBinsLog2 ? shift - kSelBinsLog2 : 0;
#pragma unroll
        for (int u = 0; u < kPer; ++u)
          if (key[u]) atomicAdd(&hist[(key[u] - lo) >> coarse], 1u);
        __syncthreads();
        uint32_t all;
        uint32_t b = my_bin(hist);
        place_rank(b, count_above_mine(b, s_warp, &all), a.k - n_above, s_res);
        __syncthreads();
        tau = lo + (s_res[0] << coarse);
        n_greater = n_above + s_res[1];
        if (coarse) {
#pragma unroll
          for (int u = 0; u < kPer; ++u)
            if (key[u] >= tau && ((key[u] - tau) >> coarse) == 0u) atomicAdd(&hist[kSelBins + key[u] - tau], 1u);
          __syncthreads();
          b = my_bin(hist + kSelBins);
          place_rank(b, count_above_mine(b, s_warp, &all), a.k - n_greater, s_res + 3);
          __syncthreads();
          tau += s_res[3];
          n_greater += s_res[4];
        }
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
          if (key[u] > tau) atomicAdd(&nk[kSelMaxCtas + who[u]], 1u);
          else if (key[u] == tau) atomicAdd(&nk[2 * kSelMaxCtas + who[u]], 1u);
        }
        __syncthreads();
        if (tid < G)
          v = ((v >> 32 << 32) + (static_cast<unsigned long long>(nk[kSelMaxCtas + tid]) << 32)) | nk[2 * kSelMaxCtas + tid];
      }
    }
    // exclusive scan over the CTAs
    const unsigned long long incl = warp_incl_u64(v);
    if (lane == 31) s_warp64[warp] = incl;
    __syncthreads();
    const unsigned long long upto = warp_incl_u64(lane < kWarps ? s_warp64[lane] : 0ull);
    const unsigned long long all = __shfl_sync(kFull, upto, 31);
    const unsigned long long base = warp ? __shfl_sync(kFull, upto, warp - 1) : 0ull;
    const bool nz = a.drop_zeros && tau == 0u;   // store variant without kept zeros
    const long long quota = nz ? 0 : static_cast<long long>(a.k) - n_greater;
    const long long n_stored = nz ? static_cast<long long>(n_greater) : static_cast<long long>(a.k);
    const long long eq_all = static_cast<long long>(all & 0xFFFFFFFFull);
    // self-check: offsets taken from wrong counts could point past the end of `values`, so nothing
    // is stored then
    const bool sound = static_cast<long long>(all >> 32) == n_greater && quota >= 0 &&
                       n_greater + (eq_all < quota ? eq_all : quota) == n_stored;
    const uint32_t verdict = again ? 1u : (sound ? 0u : 2u);
    if (step == kKeys) {                         // (the cleared words of a further round)
      if (tid == 0) fence_gpu();
      __syncthreads();
    }
    if (tid < G) word_store(a.answer + phase * (kSelMaxCtas + 2) + 2 + tid, a.token, base + incl - v);
    if (tid == 0) {
      word_store(a.answer + phase * (kSelMaxCtas + 2), a.token, tau | (static_cast<unsigned long long>(n_greater) << 32));
      word_store(a.answer + phase * (kSelMaxCtas + 2) + 1, a.token, verdict);
      if (verdict == 0u) {
        a.hdr->threshold_key = tau;
        a.hdr->n_keep = n_stored;
        a.hdr->n_greater = n_greater;
        a.hdr->tie_quota = quota;
        a.offsets[(a.n + SURGEON_BLOCK - 1) >> kBlockShift] = static_cast<uint32_t>(n_stored);   // the sentinel entry
      } else if (verdict == 2u) {
        atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_INTERNAL));
      }
    }
    before = 0;                                  // CTA 0's chunks are the first
    if (verdict == 2u) return;
  } else {
    __shared__ unsigned long long s_last[3];
    if (tid < 3) {
      unsigned long long v = 0;
      const int which = tid < 2 ? tid : 2 + static_cast<int>(blockIdx.x);
      if (!word_wait(a.answer + phase * (kSelMaxCtas + 2) + which, a.token, &v)) s_fail = 1;
      s_last[tid] = v;
    }
    __syncthreads();
    if (s_fail) { quit(); return; }
    if (s_last[1] == 2ull) return;
    again = s_last[1] == 1ull;
    tau = static_cast<uint32_t>(s_last[0]);
    n_greater = static_cast<uint32_t>(s_last[0] >> 32);
    before = s_last[2];
  }
  ++phase;
  if (!again) break;
  step = kRefine;
  }
  const bool nz = a.drop_zeros && tau == 0u;     // store variant without kept zeros
  const long long quota = nz ? 0 : static_cast<long long>(a.k) - n_greater;
  const long long n_stored = nz ? static_cast<long long>(n_greater) : static_cast<long long>(a.k);

  // ---- per-chunk counts and places ----
  if (step == kKeys) {                           // what was above the bin, and the CTA's few keys inside it
    const int n_bin = static_cast<int>(s_nkeys);
    for (int c = tid; c < n_local; c += kThreads) {
      uint32_t both = static_cast<uint32_t>(prefix[c]);
#pragma unroll 1
      for (int i = 0; i < n_bin; ++i)
        if (s_bin_chunk[i] == c && s_bin_key[i] >= tau) both += s_bin_key[i] > tau ? 1u : 0x10000u;
      cnt[c] = both;
    }
    __syncthreads();
  }
  unsigned long long carry = before;
  constexpr int kScan = 4;                       // consecutive chunks per thread
  for (int c0 = 0; c0 < n_local; c0 += kScan * kThreads) {
    const int c = c0 + kScan * tid;
    unsigned long long val[kScan], sum = 0;
#pragma unroll
    for (int j = 0; j < kScan; ++j) {
      const uint32_t v = c + j < n_local ? cnt[c + j] : 0u;
      val[j] = (static_cast<unsigned long long>(v & 0xFFFFu) << 32) | (v >> 16);
      sum += val[j];
    }
    const unsigned long long incl = warp_incl_u64(sum);
    if (lane == 31) s_warp64[warp] = incl;
    __syncthreads();
    const unsigned long long upto = warp_incl_u64(lane < kWarps ? s_warp64[lane] : 0ull);
    unsigned long long base = carry + incl - sum + (warp ? __shfl_sync(kFull, upto, warp - 1) : 0ull);
    carry += __shfl_sync(kFull, upto, 31);
#pragma unroll
    for (int j = 0; j < kScan; ++j) {
      if (c + j < n_local) prefix[c + j] = base;
      base += val[j];
    }
    __syncthreads();
  }

  // ---- emit ----
  unsigned char* stage = aux + warp * kStageBytes;
  auto emit = [&](int c, unsigned char* region) -> bool {
    const unsigned long long at = prefix[c - c_begin];
    return emit_chunk<DT>(a, region, stage, c, tau, quota, at, cnt[c - c_begin] >> 16, n_stored);
  };
  if (RES) {
    run_resident(false, emit);
  } else if (spread) {
    if (!meet()) { quit(); return; }             // every CTA's places are known to all
    tc::fence_proxy_async();
    __syncwarp();
    begin_pass(true);                            // from the end, where the L2 cache holds some of it
    unsigned long long at_next = fly0 < a.n_chunks ? prefix[fly0 - c_begin] : 0ull;    // fetched one chunk ahead
    uint32_t n_next = fly0 < a.n_chunks ? cnt[fly0 - c_begin] : 0u;
    run_pass(true, [&](int c, unsigned char* region) -> bool {
      const unsigned long long at = at_next;
      const uint32_t n_at = n_next >> 16;
      if (fly1 < a.n_chunks) { at_next = prefix[fly1 - c_begin]; n_next = cnt[fly1 - c_begin]; }
      return emit_chunk<DT>(a, region, stage, c, tau, quota, at, n_at, n_stored);
    });
    if (s_fail && lane == 0) atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
  } else {
    // the chunks still in the ring first, then backwards through the rest
    for (int i = n_mine - 1; i >= 0; --i) {
      const int sl = i % kSlotsPerWarp;
      if (i + kSlotsPerWarp < n_mine && !arrived(chunk_of(i), sl)) {
        atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
        for (int j = i - 1; j >= 0 && j > i - kSlotsPerWarp; --j) arrived(chunk_of(j), j % kSlotsPerWarp);
        break;
      }
      const bool written = emit(chunk_of(i), my_ring + sl * kChunkBytes);
      if (i >= kSlotsPerWarp) {
        if (written) tc::fence_proxy_async();
        __syncwarp();
        issue(chunk_of(i - kSlotsPerWarp), sl);
      }
    }
  }
}

// n_keep == 0 (ratio 1, or an empty tensor): nothing to select.
__global__ void header_empty_kernel(surgeon_header* hdr, uint32_t sentinel, uint32_t* offsets,
                                    long long n_blocks) {
  offsets[n_blocks] = 0u;                        // the sentinel entry of the block offsets
  hdr->threshold_key = sentinel;
  hdr->status = SURGEON_OK;
  hdr->n_keep = 0;
  hdr->n_greater = 0;
  hdr->tie_quota = 0;
}

// ---- decompress -------------------------------------------------------------------------------
// Algorithm 1, Reshape step: one warp rebuilds 1024 elements (32 bitmap words) of the dense tensor.
// The piece's packed values are one contiguous run: they are staged in shared memory with 16-byte
// loads; a lane then puts the values of its bitmap word (a loop over the set bits, about 8
// instructions per kept element of the fullest word) into its row of a zeroed tile, and the tile
// leaves as 16-byte vectors.  Bound by the memory; a lane per element, with two-byte stores and two
// shuffles and a population count each, took 53 us on 38.7 M bf16 elements (ratio 0.7), this 45.
constexpr int kDecWarps = 8;
constexpr int kDecElems = 1024;
template <int DT>
__host__ __device__ constexpr int dec_warp_bytes() {                 // the tile, and the values with alignment slack
  return 2 * kDecElems * static_cast<int>(sizeof(typename Elem<DT>::type)) + 32;
}
template <int DT>
__global__ void __launch_bounds__(kDecWarps * 32)
decompress_kernel(const uint32_t* __restrict__ bitmap, const void* __restrict__ values_v,
                  const uint32_t* __restrict__ offsets, long long n, void* __restrict__ out_v) {
  using E = typename Elem<DT>::type;
  constexpr int EPV = 16 / sizeof(E);
  constexpr int kRowVecs = 32 / EPV;             // 16-byte vectors of a lane's row: 8 / 4
  const E* __restrict__ values = reinterpret_cast<const E*>(values_v);
  E* __restrict__ out = reinterpret_cast<E*>(out_v);
  extern __shared__ __align__(128) unsigned char dec_smem[];
  unsigned char* tile = dec_smem + (threadIdx.x >> 5) * dec_warp_bytes<DT>();
  E* stage = reinterpret_cast<E*>(tile + kDecElems * sizeof(E));
  const uint32_t lane = lane_id();
  // vectors of a row are XORed with the row's number: lanes at the same place of their rows differ in banks
  auto swz = [](uint32_t row) { return DT == 0 ? (row & 7u) : ((row >> 1) & 3u); };
  const long long n_chunks = (n + kDecElems - 1) / kDecElems;
  const long long n_words = (n + 31) / 32;
  const long long n_blocks = (n + SURGEON_BLOCK - 1) >> kBlockShift;
  const long long warps = (static_cast<long long>(gridDim.x) * blockDim.x) >> 5;
  const uint32_t n_vals = offsets[n_blocks];
  for (long long chunk = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
       chunk < n_chunks; chunk += warps) {
    const long long w_idx = chunk * 32 + lane;
    uint32_t word = (w_idx < n_words) ? bitmap[w_idx] : 0u;
    const uint32_t first = offsets[chunk * (kDecElems / SURGEON_BLOCK)];
    const uint32_t cnt = __popc(word);
    const uint32_t excl = warp_excl_scan(cnt);
    const uint32_t total = __shfl_sync(kFull, excl + cnt, 31);
    // the values, from the vector that holds the first one on
    const uint32_t a0 = first & ~static_cast<uint32_t>(EPV - 1);
    const uint32_t n_vec = total ? (first + total - a0 + EPV - 1) / EPV : 0u;
    for (uint32_t v = lane; v < n_vec; v += 32) {
      const uint32_t e0 = a0 + v * EPV;
      if (e0 + EPV <= n_vals) {
        reinterpret_cast<uint4*>(stage)[v] = __ldg(reinterpret_cast<const uint4*>(values + e0));
      } else {                                   // the vector that ends past the last value
        for (uint32_t e = 0; e < static_cast<uint32_t>(EPV) && e0 + e < n_vals; ++e) stage[v * EPV + e] = values[e0 + e];
      }
    }
    unsigned char* row = tile + lane * (32 * sizeof(E));
#pragma unroll
    for (int j = 0; j < kRowVecs; ++j) reinterpret_cast<uint4*>(row)[j] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    const E* src = stage + (first - a0) + excl;
    while (word) {
      const uint32_t e = __ffs(word) - 1;
      word &= word - 1;
      const uint32_t byte = e * static_cast<uint32_t>(sizeof(E));
      *reinterpret_cast<E*>(row + (((byte >> 4) ^ swz(lane)) << 4) + (byte & 15u)) = *src++;
    }
    __syncwarp();
    const long long base = chunk * kDecElems;
#pragma unroll
    for (int j = 0; j < kRowVecs; ++j) {
      const uint32_t v = j * 32 + lane, r = v / kRowVecs, c = v % kRowVecs;
      const uint4 q = *reinterpret_cast<const uint4*>(tile + r * (32 * sizeof(E)) + ((c ^ swz(r)) << 4));
      const long long idx = base + v * EPV;
      if (idx + EPV <= n) {
        *reinterpret_cast<uint4*>(out + idx) = q;
      } else {
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int e = 0; e < EPV; ++e)
          if (idx + e < n) out[idx + e] = static_cast<E>((DT == 0) ? w[e % 4] : (w[e >> 1] >> (16 * (e & 1))));
      }
    }
    __syncwarp();                                // the tile and the stage are the next piece's
  }
}

using TmaEncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                 const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                 const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The tensor as rows of 128 bytes (32 words), box = one chunk, 128-byte swizzle.
bool make_row_map(const void* x, long long n_rows_full, CUtensorMap* map) {
  const TmaEncodeFn encode = reinterpret_cast<TmaEncodeFn>(tensor_map_encode_fn());
  if (!encode) return false;
  const cuuint64_t dims[2] = {32, static_cast<cuuint64_t>(n_rows_full)};
  const cuuint64_t strides[1] = {128};
  const cuuint32_t box[2] = {32, 32};
  const cuuint32_t estr[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<void*>(x), dims, strides, box,
                estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// A value that no other call of this or another process carries (see the grid-wide exchange).
unsigned long long next_token() {
  static std::atomic<unsigned long long> counter{[] {
    std::random_device rd;
    const unsigned long long t = static_cast<unsigned long long>(
        std::chrono::steady_clock::now().time_since_epoch().count());
    return ((static_cast<unsigned long long>(rd()) << 32) | rd()) ^ (t << 20);
  }()};
  unsigned long long v = counter.fetch_add(1, std::memory_order_relaxed);
  return v ? v : counter.fetch_add(1, std::memory_order_relaxed);
}

template <int DT>
cudaError_t run_prune_compact(const void* x, long long n, long long k, int drop_zeros, int stall, int share,
                              const surgeon_compressed& out, void* workspace,
                              cudaStream_t stream) {
  using E = typename Elem<DT>::type;
  if (k == 0) {
    const long long n_blocks = (n + SURGEON_BLOCK - 1) >> kBlockShift;
    if (n > 0) {   // nothing is kept: an empty bitmap, and no value before any block
      cudaError_t e = cudaMemsetAsync(out.bitmap, 0, static_cast<size_t>((n + 31) / 32) * 4, stream);
      if (e == cudaSuccess) e = cudaMemsetAsync(out.block_offsets, 0, static_cast<size_t>(n_blocks) * 4, stream);
      if (e != cudaSuccess) return e;
    }
    header_empty_kernel<<<1, 1, 0, stream>>>(out.header, Elem<DT>::kSentinel, out.block_offsets, n_blocks);
    note_launches(1);
    return cudaGetLastError();
  }
  const PruneLayout L = prune_layout(n, DT);
  char* ws = static_cast<char*>(workspace);
  PruneArgs a;
  a.x = x; a.n = n; a.k = static_cast<uint32_t>(k);
  a.n_rows_full = n * static_cast<long long>(sizeof(E)) / 128;
  a.n_chunks = static_cast<int>(L.tiles);
  a.drop_zeros = drop_zeros; a.stall = stall;
  a.token = next_token();
  a.hdr = out.header; a.bitmap = out.bitmap; a.values = out.values; a.offsets = out.block_offsets;
  a.arrive = reinterpret_cast<ulonglong2*>(ws + L.arrive);
  a.answer = reinterpret_cast<ulonglong2*>(ws + L.answer);
  a.keys = reinterpret_cast<uint32_t*>(ws + L.keys);
  a.hist = reinterpret_cast<uint32_t*>(ws + L.hist);
  a.claims = reinterpret_cast<uint32_t*>(ws + L.claims);
  a.cnt = reinterpret_cast<uint32_t*>(ws + L.cnt);
  a.prefix = reinterpret_cast<unsigned long long*>(ws + L.prefix);
  a.slots = ws + L.slots;
  CUtensorMap map;
  if (!make_row_map(x, a.n_rows_full > 0 ? a.n_rows_full : 1, &map)) return cudaErrorNotSupported;
  // A call by itself: as many chunks per warp as a full grid would give its busiest warp, on as few CTAs as that
  // takes.  A CTA takes a whole SM, so calls on full grids run one after the other, each with its chain of exchanges
  // exposed (20 us of the 40 that 19 MB take).  A call that says that others run beside it (SURGEON_SHARE_GPU) gets
  // the smallest grid that keeps the tensor on chip, and of a tensor that no quarter of the SMs can hold a
  // quarter: four such grids fit exactly (of grids that leave a rest a fifth starts in part and spins).
  // Whole stacks on eight streams, full grid / SMs / 2, / 3, / 4: ViT 2.46 / 1.70 / 1.57 / 1.61 ms, WideResNet
  // 1.53 / 1.14 / 1.08 / 0.96, ResNet-50 1.68 / 1.28 / 1.09 / 1.02, ResNeXt 1.93 / 1.46 / 1.36 / 1.24.
  const int sms = sm_count() < kSelMaxCtas ? sm_count() : kSelMaxCtas;
  int grid;
  if (share) {
    const int most = std::min(sms, std::max(sms / 4, kLeastStreamedCtas));
    grid = std::min(most, (a.n_chunks + kResidentChunks - 1) / kResidentChunks);
  } else {
    const int per_cta = (a.n_chunks + sms * kWarps - 1) / (sms * kWarps) * kWarps;
    grid = (a.n_chunks + per_cta - 1) / per_cta;
  }
  // claimed chunks (see the kernel): by itself from 512 chunks per CTA on, where equal shares end unevenly; on a part
  // of the GPU only where the counts do not fit (on a quarter, 131 MB: 335 -> 310 us bf16, 260 -> 238 fp32)
  a.spread = a.n_chunks > grid * (share ? kMaxLocalChunks : 512) ? 1 : 0;
  const bool resident = (a.n_chunks + grid - 1) / grid <= kResidentChunks;
  const void* kernel = resident ? reinterpret_cast<const void*>(prune_kernel<DT, true>)
                                : reinterpret_cast<const void*>(prune_kernel<DT, false>);
  cudaError_t e = allow_dynamic_smem(kernel, static_cast<int>(kPruneSmem));
  if (e != cudaSuccess) return e;
  void* args[] = {&map, &a};
  e = cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(kThreads), args, kPruneSmem, stream);
  if (e != cudaSuccess) return e;
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_prune_compact(const void* x, int64_t n, int dt, int64_t k,
                                 const surgeon_compressed& out, void* workspace,
                                 cudaStream_t stream, int drop_zeros, int stall, int share) {
  return dt == 0 ? run_prune_compact<0>(x, n, k, drop_zeros, stall, share, out, workspace, stream)
                 : run_prune_compact<1>(x, n, k, drop_zeros, stall, share, out, workspace, stream);
}

cudaError_t launch_decompress(const surgeon_compressed& act, void* x_out, cudaStream_t stream) {
  if (act.n == 0) return cudaSuccess;
  const long long n_chunks = (act.n + kDecElems - 1) / kDecElems;
  const long long ctas = (n_chunks + kDecWarps - 1) / kDecWarps;
  // a few pieces per warp of a full device (six CTAs per SM in bf16, three in fp32)
  const long long cap = 4LL * (act.dt == 0 ? 3 : 6) * sm_count();
  const int grid = static_cast<int>(ctas < cap ? ctas : cap);
  auto launch = [&](auto kernel, int bytes) -> cudaError_t {
    const cudaError_t e = allow_dynamic_smem(reinterpret_cast<const void*>(kernel), bytes);
    if (e != cudaSuccess) return e;
    kernel<<<grid, kDecWarps * 32, bytes, stream>>>(act.bitmap, act.values, act.block_offsets, act.n, x_out);
    note_launches(1);
    return cudaGetLastError();
  };
  return act.dt == 0 ? launch(decompress_kernel<0>, kDecWarps * dec_warp_bytes<0>())
                     : launch(decompress_kernel<1>, kDecWarps * dec_warp_bytes<1>());
}

}  // namespace surgeon
