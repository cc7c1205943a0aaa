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
//             overwhelming probability (1-6 % of the elements)
//   classify  first pass over the CTA's chunks: keys above the bracket are counted per chunk, the
//             keys inside are listed and counted in a histogram of 512 bins over the bracket
//   exchange  the summed histogram gives the threshold's bin: one key for bf16, whose brackets are
//             narrower than 512 keys, some thousands of keys for fp32, of which few occur
//   exchange  every CTA reports its count above the bin and the keys it has inside; CTA 0 finds the
//             threshold among them and gives every CTA its place in the packed vector.  Where the bin is one key
//             (bf16; one key everywhere; a threshold of zero) there is none: every CTA has shown the others what it has
//             above each bin and in it, and adds up for itself what lies before it.  2^20 bf16 18.5 -> 16.5 us, 2^23
//             24.3 -> 22.6, 77 MB 63.5 -> 61.5
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
#include <type_traits>

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
// The rest of the shared memory: 32 KB, all of it the sample's bins first.
constexpr int kMaxLocalChunks = 1024;            // per-chunk counts in shared memory up to here
constexpr int kSampleBinsLog2 = 14;              // top 14 key bits: 64 bins per octave; 16-bit counters here
constexpr int kAuxBytes = 2 << kSampleBinsLog2;
static_assert((1 << kSampleBinsLog2) == kSampleBins, "bins of the sample");
constexpr int kAuxSlots = 8192;                  // (histograms before it)
// A resident range: the listed keys of a chunk have a slot of their own, 12 % of its elements.
constexpr int kResSlotBytes = 496;
constexpr int kResCnt = kAuxSlots + kResidentChunks * kResSlotBytes;
constexpr int kResPrefix = kResCnt + kResidentChunks * 4;
static_assert(kResPrefix % 8 == 0 && kResPrefix + kResidentChunks * 8 <= kAuxBytes, "shared memory of a resident range");
// Others: a staging slot per warp (room for 1/16 of a chunk), and one list of the keys of all chunks, each chunk's
// in one piece.  What does not fit there goes to the chunk's slot in global memory.  The places take the list's room when
// it is done with.
constexpr int kSlotBytes = 256;
constexpr int kListStart = kAuxSlots + kWarps * kSlotBytes;          // where a chunk's keys begin, 16 bits
constexpr int kListAcc = kListStart + kMaxLocalChunks * 2;           // its count above the bin, 16 bits
constexpr int kList = kListAcc + kMaxLocalChunks * 2;
constexpr int kListBytes = 12288;
// Counts and places of the chunks that there are lie at the end.
static_assert(kList + kListBytes + kMaxLocalChunks * 4 <= kAuxBytes, "shared memory of a streamed range");
constexpr size_t kPruneSmem = static_cast<size_t>(kRingBytes) + kAuxBytes + 1024;
static_assert(kChunkBytes == kTileVecs * 16, "chunk size");
// A streamed tensor's bracket comes from order statistics 2.5 sqrt(G) + 1 places to either side of the middle of G
// CTAs' answers: with fewer than 31 CTAs there are none, and every key would be a candidate.
constexpr int kLeastStreamedCtas = 31;
constexpr int kMaxKeys = 64;                     // keys one CTA reports at the last exchange, where the scratch has room
constexpr uint32_t kKeysAtOnce = 960;            // and CTA 0 takes in, two threads per CTA
static_assert(2 * kSelMaxCtas <= kThreads && kSelMaxCtas <= 256 &&
              4 * (kSelBins + kKeysAtOnce + kSelMaxCtas) + kKeysAtOnce <= kAuxSlots, "room of the keys at CTA 0");

struct PruneArgs {
  const void* x;
  long long n, n_rows_full;      // elements; whole 128-byte rows (what the tensor map covers)
  uint32_t k;
  int n_chunks;                  // chunks in all
  int drop_zeros, stall;
  unsigned long long token;      // unlike any other call's
  unsigned long long table_base; // the table's tag: unlike any other call's; (replayed) any other process's
  int replayed;                  // the call is captured: its executions are counted
  surgeon_header* hdr;
  uint32_t* bitmap;
  void* values;
  uint32_t* offsets;
  ulonglong2* arrive;            // [kSelPhases][kSelMaxCtas]: {token, what the CTA reports}
  ulonglong2* answer;            // [kSelPhases][kSelMaxCtas + 2]: {token, what CTA 0 answers}
  unsigned long long* keys;      // [CTAs][key_room()]: {tag, key}
  uint32_t* hist;                // [kSelHists][kSelBins]
  uint32_t* claims;              // [kSelPhases][kClaimSets], kClaimStride words apart: groups claimed in each pass
  uint32_t* cnt;                 // per chunk (kClaimed)
  unsigned long long* prefix;    // likewise
  ulonglong2* table;             // [CTAs][table_bins()]: {tag, counts above the bin and (lower half) inside}
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
// No word has to start at zero, so the call needs no memset: the token differs from call to
// call.  For a captured graph, whose replays carry the same token, CTA 0 clears every report that it
// has read, clears the answers of the phases to come before an answer that leads to them, and clears that of phase 0
// after the reports of phase 1; a CTA takes its words back when it gives up.
// All CTAs are resident (cooperative launch); polls are bounded.
//
// No fence stands between a report and the answer: one waits for the stores before it, 0.3-0.5 us, and an exchange
// used to have four of them in its chain.  Keys carry a tag each, so they are polled like the words; the
// bins, which are added up by atomics, are complete when their sum is the sum of the counts in the words.  (148 CTAs:
// words alone 1.3 us, with atomics behind fences 4.1; measured on exchanges alone.)
//
// A tag is 32 bits, which something that the scratch happens to hold, or that an earlier replay left there, could match.
// So every CTA clears its key words before the fence that precedes its first report, and CTA 0 has a fence behind
// these reports where it asks for keys, off the chain (it has answered by then): it sees cleared words or this call's.
// Where a CTA has more keys than it can report, the bin is narrowed and keys are reported once more, in the same words: the
// tag names the phase.
//
// The table's words are not cleared (every CTA reads those of all others, so a fence would stand in every CTA's chain).
// Their tag is 64 bits.  A call that is launched has one of its own, like its token.  Of a captured call, which may run many times,
// it is the process's random number and how many such executions the GPU has begun: CTA 0 counts them and tells the others with its
// first answer.  No two executions have the same.  (Counted always, calls on 2^15 to 2^26 elements took 1.3 % longer.)
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
// (never that of a cleared word)
__device__ __forceinline__ uint32_t key_tag(unsigned long long token, int phase) {
  return (static_cast<uint32_t>(token) << 4) | static_cast<uint32_t>(phase);
}
static_assert(kSelPhases <= 16, "phase in four bits");
__device__ __forceinline__ void key_store(unsigned long long* p, uint32_t tag, uint32_t key) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"((static_cast<unsigned long long>(tag) << 32) | key) : "memory");
}
// (not wanted: the tag and `otherwise`)
__device__ __forceinline__ unsigned long long key_load_if(const unsigned long long* p, bool wanted, uint32_t tag, uint32_t otherwise) {
  unsigned long long v = (static_cast<unsigned long long>(tag) << 32) | otherwise;
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.relaxed.gpu.global.u64 %0, [%1];\n\t}"
               : "+l"(v) : "l"(p), "r"(static_cast<uint32_t>(wanted)) : "memory");
  return v;
}
// Executions of the kernel on this GPU so far (at most 2^64): part of the tags of the table, see below.
__device__ unsigned long long g_executions;
__device__ __forceinline__ uint32_t count_load(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ int key_room(int ctas) { return min(kMaxKeys, kSelMaxCtas * kMaxKeys / 2 / ctas); }
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// One thread waits for a word of this call (what it announces apart from its own 8 bytes is visible
// after a fence).  `stall` is the diagnostic of SURGEON_DEBUG_STALL_BARRIER: a value nobody ever
// stores, and a cap of 1024 polls.
__device__ __forceinline__ bool word_wait(const ulonglong2* p, unsigned long long token, unsigned long long* v,
                                          bool stall = false) {
  const uint32_t cap = stall ? 1024u : (1u << 22);
#pragma unroll 1
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

// put(which, value) for the elements of this lane's row whose bits are set; `which` = rank among them.  U elements of
// each word per turn, so that their loads overlap: a turn is a chain of a bit search, a load and a store, 170 clocks.
template <int DT, int WPL, int U, typename F>
__device__ __forceinline__ void take_set(const unsigned char* region, const uint32_t (&word)[WPL], F put) {
  using E = typename Elem<DT>::type;
  const uint32_t lane = lane_id(), x = (lane & 7) << 4;
  const unsigned char* row = region + lane * 128;
  uint32_t m[WPL], at[WPL];
#pragma unroll
  for (int w = 0; w < WPL; ++w) {
    m[w] = word[w];
    at[w] = w ? __popc(word[0]) : 0u;
  }
#pragma unroll 1
  while (m[0] | m[WPL - 1]) {
    E val[WPL][U];
    bool have[WPL][U];
#pragma unroll
    for (int w = 0; w < WPL; ++w) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        have[w][u] = m[w] != 0u;
        const uint32_t e = 32 * w + (__clz(__brev(m[w])) & 31);      // (no bit left: some element of the row)
        m[w] &= m[w] - 1u;
        val[w][u] = *reinterpret_cast<const E*>(row + ((e * static_cast<uint32_t>(sizeof(E))) ^ x));
      }
    }
#pragma unroll
    for (int w = 0; w < WPL; ++w) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (have[w][u]) put(at[w] + u, val[w][u]);
      at[w] += U;
    }
  }
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

// Keys of the chunk above t, and (upper half) equal to it.
template <int DT>
__device__ __noinline__ uint32_t count_chunk(const unsigned char* region, uint32_t t) {
  constexpr int EPR = 128 / static_cast<int>(sizeof(typename Elem<DT>::type)), WPL = EPR / 32;
  uint4 q[8];
  load_row(region, q);
  uint32_t m[WPL], ge = 0, gt = 0;               // (t >= 1: what lies past the tensor's end is below it)
  mask_ge<DT, WPL>(q, EPR, t, m);
#pragma unroll
  for (int w = 0; w < WPL; ++w) ge += __popc(m[w]);
  mask_ge<DT, WPL>(q, EPR, t + 1u, m);
#pragma unroll
  for (int w = 0; w < WPL; ++w) gt += __popc(m[w]);
  return __reduce_add_sync(kFull, gt | ((ge - gt) << 16));
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

// The bits of a row in the one chunk inside which the tie quota ends: `above` and the first `allowed` ties of the chunk, which
// are ranked by flat index (= lane, then bit).  Out of line, like all that one chunk of a tensor does: code that is not
// in the instruction caches costs some 250 clocks per 128 bytes, and a call runs most of its code once.
template <int DT>
__device__ __noinline__ uint2 quota_words(const unsigned char* region, int nv, uint32_t tau, long long allowed, uint2 above) {
  constexpr int WPL = 128 / static_cast<int>(sizeof(typename Elem<DT>::type)) / 32;
  uint4 q[8];
  load_row(region, q);
  uint32_t word[2] = {above.x, above.y}, ge[WPL], ec = 0;
  mask_ge<DT, WPL>(q, nv, tau, ge);
#pragma unroll
  for (int w = 0; w < WPL; ++w) { ge[w] &= ~word[w]; ec += __popc(ge[w]); }
  allowed -= warp_excl_scan(ec);
#pragma unroll
  for (int w = 0; w < WPL; ++w) {
    word[w] |= lowest_set_bits(ge[w], allowed);
    allowed -= __popc(ge[w]);
  }
  return make_uint2(word[0], word[1]);
}

// The byte at address a of a packed sequence lives at a ^ ((a >> 5) & 0x7C): the 32-bit word
// index is XORed with the index of its 128-byte row.  Without it, lanes that keep their whole
// row (chunks before the end of a large tie quota, e.g. the zeros of post-ReLU data at a low
// ratio) all start a multiple of 32 words apart and every store of the gather is a 32-way
// bank conflict.
__device__ __forceinline__ uint32_t packed_at(uint32_t addr) { return addr ^ ((addr >> 5) & 0x7Cu); }
template <int DT>
__device__ __forceinline__ uint32_t packed_elem(uint32_t rbase, uint32_t i) {        // element i of the sequence
  const uint32_t addr = packed_at(rbase + i * static_cast<uint32_t>(sizeof(typename Elem<DT>::type)));
  uint32_t u;
  unsigned short h;
  if (DT == 0) { asm volatile("ld.shared.u32 %0, [%1];" : "=r"(u) : "r"(addr) : "memory"); return u; }
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(h) : "r"(addr) : "memory");
  return h;
}
// A full chunk with a misaligned destination: no room for the shift, the vectors are put together from elements.
template <int DT>
__device__ __noinline__ void copy_full_chunk(typename Elem<DT>::type* values, long long kept_before, uint32_t total, uint32_t rbase,
                                             long long n_stored, uint32_t* status) {
  using E = typename Elem<DT>::type;
  constexpr int EPV = 16 / sizeof(E);
  const uint32_t lane = lane_id(), mis = static_cast<uint32_t>(kept_before % EPV);
  E* dst = values + kept_before;
  const uint32_t head = min(mis ? EPV - mis : 0u, total);
  const uint32_t n_vec = (total - head) / EPV;
  if (lane < head && SURGEON_IN_BOUNDS(kept_before + lane, n_stored, status))
    dst[lane] = static_cast<E>(packed_elem<DT>(rbase, lane));
#pragma unroll 1
  for (uint32_t v = lane; v < n_vec; v += 32) {
    const uint32_t b = head + v * EPV;
    uint32_t o[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      o[i] = DT == 0 ? packed_elem<DT>(rbase, b + i)
                     : packed_elem<DT>(rbase, b + 2 * i) | (packed_elem<DT>(rbase, b + 2 * i + 1) << 16);
    if (SURGEON_IN_BOUNDS(kept_before + head + v * EPV + EPV - 1, n_stored, status))
      *reinterpret_cast<uint4*>(dst + head + v * EPV) = make_uint4(o[0], o[1], o[2], o[3]);
  }
  const uint32_t done = head + n_vec * EPV;
  if (lane < total - done && SURGEON_IN_BOUNDS(kept_before + done + lane, n_stored, status))
    dst[done + lane] = static_cast<E>(packed_elem<DT>(rbase, done + lane));
}

// ---- emit one chunk -------------------------------------------------------------------------------
// before = (elements above the threshold before the chunk) << 32 | (ties before it); n_eq = its ties.
// True when the chunk's place in the ring has been written to.
template <int DT>
__device__ __forceinline__ bool emit_chunk(const PruneArgs& a, unsigned char* region, int chunk, uint32_t tau, long long quota,
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
    const uint2 above = make_uint2(word[0], word[WPL - 1]);
    const uint2 both = quota_words<DT>(region, nv, tau, quota - eq_b, above);
    word[0] = both.x;
    if (WPL == 2) word[WPL - 1] = both.y;
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
  // Gathered in place in the chunk's own part of the ring, whatever share is kept.  (Sparse chunks by a loop over the set
  // bits into a staging area took as long where 7-10 % are kept, and longer elsewhere: bf16, 77 MB, 30 % kept 72 against
  // 65.5 us, 537 MB 353 against 314.)
  __syncwarp();                                  // every lane has its row in registers
  const uint32_t rbase = smem_u32(region);
  const bool lined_up = total + mis <= static_cast<uint32_t>(32 * EPR);
  uint32_t pa = rbase + (lane_pre + (lined_up ? mis : 0u)) * static_cast<uint32_t>(sizeof(E));
  auto gather = [&](auto at) {
    auto put = [&](uint32_t v) {
      if (DT == 0) asm volatile("st.shared.u32 [%0], %1;" ::"r"(at(pa)), "r"(v) : "memory");
      else asm volatile("st.shared.u16 [%0], %1;" ::"r"(at(pa)), "h"(static_cast<unsigned short>(v)) : "memory");
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
  };
  // Rows kept by five eighths at most start far enough from multiples of 32 words without the XOR, which is a third
  // of the gather's instructions: bf16, 2 GB, a tenth kept 980 -> 920 us, 537 MB 292 -> 274, 77 MB 65.5 -> 63.5; fp32,
  // 131 MB 84.0 -> 81.9, 4.3 GB, a tenth kept 1562 -> 1514 (half kept: 1857 and 1856, runs of one side differ by 20).
  constexpr uint32_t kMost = 5u * EPR / 8u;
  if (lined_up && total <= 32u * kMost && __reduce_max_sync(kFull, cnt) <= kMost) {
    gather([](uint32_t addr) { return addr; });
    __syncwarp();
    E* gbase = values + (kept_before - mis);
    const uint32_t end = mis + total, v_first = mis ? 1u : 0u, v_end = end / EPV;
    const E* packed = reinterpret_cast<const E*>(region);
    const uint32_t tail = (v_end > v_first ? v_end : v_first) * EPV;
    if (mis && mis + lane < static_cast<uint32_t>(EPV) && mis + lane < end &&
        SURGEON_IN_BOUNDS(kept_before + lane, n_stored, &a.hdr->status))
      gbase[mis + lane] = packed[mis + lane];
    if (tail + lane < end && SURGEON_IN_BOUNDS(kept_before - mis + tail + lane, n_stored, &a.hdr->status))
      gbase[tail + lane] = packed[tail + lane];
#pragma unroll 4
    for (uint32_t g = v_first + lane; g < v_end; g += 32)
      if (SURGEON_IN_BOUNDS(kept_before - mis + g * EPV + EPV - 1, n_stored, &a.hdr->status))
        *reinterpret_cast<uint4*>(gbase + g * EPV) = *reinterpret_cast<const uint4*>(region + g * 16);
    return true;
  }
  gather([](uint32_t addr) { return packed_at(addr); });
  __syncwarp();
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
        gbase[sl] = static_cast<E>(packed_elem<DT>(rbase, sl));
    }
#pragma unroll 4
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
      gbase[t0 + lane] = static_cast<E>(packed_elem<DT>(rbase, t0 + lane));
  } else {
    copy_full_chunk<DT>(values, kept_before, total, rbase, n_stored, &a.hdr->status);
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
#pragma unroll 1
  for (uint32_t i = lane_id(); i < n_in; i += 32) f(static_cast<uint32_t>(slot[i]));
}
// Of slots in global memory: f(c, acc, key) for the listed keys of the wanted ones of chunks
// 0 .. n_local - 1, then done(c, cnt[c], the chunk's acc).  A lane per chunk, 64 bytes at a time: many chunks in
// flight, and little more asked for than the keys (half a warp per chunk made 4.3 GB 6 % slower).
template <int DT, typename W, typename F, typename D>
__device__ __forceinline__ void slot_keys_global(const typename Elem<DT>::type* slots, const uint32_t* cnt, int n_local, W wanted, F f, D done) {
  constexpr uint32_t EPV = 16 / sizeof(typename Elem<DT>::type);
#pragma unroll 1
  for (int c = threadIdx.x; c < n_local; c += kThreads) {
    if (!wanted(c)) continue;
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

// CTA 0: no phase of [p0, p1) has an answer, and the bins and counts of the rounds [r0, r1) are zero.
__device__ __forceinline__ uint32_t* above_count(const PruneArgs& a, int round) {     // (between the counters of claims)
  return a.claims + round * kClaimSets * kClaimStride + 1;
}
// Prepared before the first answer: two rounds, each with an exchange of its own and perhaps a last one.  (A round whose bins are
// cleared later begins behind fences: 131072 fp32, half of them zeros, 22.4 us and 20.9.)
constexpr int kFirstRounds = 2, kFirstPhases = 1 + 2 * kFirstRounds;
__device__ __forceinline__ void prepare_exchanges(const PruneArgs& a, int p0, int p1, int r0, int r1) {
  constexpr int kRow = kSelMaxCtas + 2;
  static_assert(kRow <= kThreads && kSelBins <= kThreads && kSelHists <= kSelPhases, "one thread per answer and bin");
  for (int p = p0; p < p1; ++p)
    if (threadIdx.x < gridDim.x + 2u) a.answer[p * kRow + threadIdx.x].x = 0ull;
  for (int r = r0; r < r1; ++r) {
    if (threadIdx.x < kSelBins) a.hist[r * kSelBins + threadIdx.x] = 0u;
    if (threadIdx.x == 0) *above_count(a, r) = 0u;
  }
}

// MODE kResident: the CTA's whole range stays in the ring (at most kResidentChunks chunks per CTA).
//      kStreamed: it goes through the ring twice; counts and lists are in shared memory.
//      kClaimed: of a gigabyte tensor the warps claim their chunks four at a time, in either pass: equal
//      shares took some SMs 620 us and others 760, and all wait for the last.  Four sets of CTAs claim
//      from counters of their own (one counter for all passes on a claim every 3 ns, too slow).  Only
//      what is counted and placed per CTA stays a contiguous range then; counts and lists are in global memory.
enum Mode { kResident = 0, kStreamed = 1, kClaimed = 2 };
template <int DT, int MODE>
__global__ void __launch_bounds__(kThreads, 1)
prune_kernel(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ PruneArgs a) {
  using E = typename Elem<DT>::type;
  constexpr bool RES = MODE == kResident, spread = MODE == kClaimed;
  constexpr uint32_t kMask = Elem<DT>::kKeyMask;
  constexpr uint32_t kKeyMax = kMask;
  constexpr int EPR = 128 / sizeof(E);
  constexpr int WPL = EPR / 32;
  constexpr int EPV = 16 / sizeof(E);
  constexpr int kSlot = RES ? kResSlotBytes / static_cast<int>(sizeof(E)) : slot_entries(DT);
  static_assert(RES || kSlot * sizeof(E) == kSlotBytes, "slot size");
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
  __shared__ uint32_t s_over, s_fail, s_nkeys, s_list_n, s_list_lo;
  __shared__ unsigned long long s_ans[2];
  __shared__ unsigned long long s_tag;         // of the table
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
  const int n_mine = warp < n_local ? (n_local - 1 - warp) / kWarps + 1 : 0;   // (not spread) chunks c_begin + warp + 16 i
  const int n_even = (n_local + 1) & ~1;         // (the places are 8 bytes each)
  uint32_t* cnt = spread ? a.cnt + c_begin : reinterpret_cast<uint32_t*>(aux + (RES ? kResCnt : kAuxBytes - 4 * n_even));
  unsigned long long* prefix =
      spread ? a.prefix + c_begin : reinterpret_cast<unsigned long long*>(aux + (RES ? kResPrefix : kAuxBytes - 12 * n_even));
  // (streamed, not claimed) the list: fp32 keys, or bf16 keys less the bracket's lower end in a byte
  using L = typename std::conditional<DT == 0, uint32_t, unsigned char>::type;
  L* list = reinterpret_cast<L*>(aux + kList);
  unsigned short* list_start = reinterpret_cast<unsigned short*>(aux + kListStart);
  unsigned short* list_acc = reinterpret_cast<unsigned short*>(aux + kListAcc);
  constexpr uint32_t kNotListed = 0xFFFFu;       // the chunk's keys are in its slot in global memory
  E* s_slots = reinterpret_cast<E*>(aux + kAuxSlots);     // RES: the chunks' slots, else a staging slot per warp
  E* g_slots = reinterpret_cast<E*>(a.slots) + static_cast<long long>(c_begin) * kSlot;
  const E* __restrict__ x = reinterpret_cast<const E*>(a.x);

  // ---- the ring: this warp's places ----
  unsigned char* my_ring = ring + warp * (kSlotsPerWarp * kChunkBytes);
  const uint32_t my_bars = smem_u32(bars + warp * kSlotsPerWarp);
  uint32_t parity = 0;                           // bit s: phase of place s's next wait
  uint32_t under_way = 0;                        // bit s: a load of place s has been started and not waited for
  auto chunk_of = [&](int i) { return c_begin + warp + kWarps * i; };
  auto issue = [&](int c, int s) {               // start the load of chunk c into place s (one lane)
    if (static_cast<long long>(c) * 32 >= a.n_rows_full) return;
    under_way |= 1u << s;
    if (lane == 0) {
      tc::mbar_arrive_expect_tx(my_bars + 8 * s, kChunkBytes);
      tc::tma_load_2d(smem_u32(my_ring + s * kChunkBytes), &xmap, 0, c * 32, my_bars + 8 * s);
    }
  };
  auto landed = [&](int s) -> bool {             // wait for the load of place s
    const uint32_t bar = my_bars + 8 * s, phase_bit = (parity >> s) & 1u;
    parity ^= 1u << s;
    under_way &= ~(1u << s);
#pragma unroll 1
    for (uint32_t i = 0; i < tc::kWaitCap; ++i)
      if (tc::mbar_try_wait(bar, phase_bit)) return true;
    return false;
  };
  auto arrived = [&](int c, int s) -> bool {     // wait for it; the tensor's last, partial row is added
    unsigned char* region = my_ring + s * kChunkBytes;
    const long long row0 = static_cast<long long>(c) * 32;
    if (row0 + 32 <= a.n_rows_full) return landed(s);
    if (row0 < a.n_rows_full) {
      if (!landed(s)) return false;
    } else {
#pragma unroll 1
      for (int v = lane; v < kChunkBytes / 16; v += 32)
        *reinterpret_cast<uint4*>(region + v * 16) = make_uint4(0, 0, 0, 0);
      tc::fence_proxy_async();                   // (these stores precede the next TMA fill of the place)
      __syncwarp();
    }
    if (a.n > a.n_rows_full * EPR) {
      const int r = static_cast<int>(a.n_rows_full - row0);       // the map fills the rows past it with zeros
#pragma unroll 1
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
  auto start = [&](bool reverse, int s) -> int { // the load of the next chunk; reverse: from the tensor's end
    int c = next();
    if (c < a.n_chunks) {
      if (reverse) c = a.n_chunks - 1 - c;
      issue(c, s);
    }
    return c;
  };
  auto begin_pass = [&](bool reverse) {          // the first three loads
    at_i = 0;
    fly0 = start(reverse, 0); fly1 = start(reverse, 1); fly2 = start(reverse, 2);
  };
  // One pass over the warp's chunks: f(chunk, region) is true where it wrote to the region.
  auto run_pass = [&](bool reverse, auto f) {
#pragma unroll 1
    for (int s = 0; fly0 < a.n_chunks; s = s == 2 ? 0 : s + 1) {
      unsigned char* region = my_ring + s * kChunkBytes;
      if (!arrived(fly0, s)) { s_fail = 1; break; }
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
#pragma unroll 1
    for (int i = 0; i < n_mine; ++i) {
      if (loading && !arrived(chunk_of(i), i)) { s_fail = 1; break; }
      f(chunk_of(i), my_ring + i * kChunkBytes);
    }
  };
  // (streamed, not claimed) f(c, acc, key) for the listed keys of every chunk, then done(c, cnt[c], the chunk's acc) on
  // one lane: eight lanes per chunk; a lane per chunk whose keys are in global memory, where that is so of two thirds or
  // more of the keys (a chain of loads for each eight keys; fp32 on a quarter of the SMs, 134 MB, 40 % kept 250 us and 233, 70 % kept
  // 266 and 252.  Where few chunks are in global memory a second loop loses: 268 MB on all SMs 139 and 142).
  auto listed_keys = [&](auto f, auto done) {
    const bool many = s_list_n > 3u * kListBytes / sizeof(L);
#pragma unroll 1
    for (int c0 = warp * 4; c0 < n_local; c0 += kWarps * 4) {
      const int c = c0 + static_cast<int>(lane >> 3);
      const uint32_t v = c < n_local ? cnt[c] : 0u, start = (v >> 16) ? list_start[c] : 0u;
      const bool later = many && start == kNotListed;
      const uint32_t n_in = later ? 0u : min(v >> 16, static_cast<uint32_t>(kSlot));
      uint32_t acc = 0;
#pragma unroll 1
      for (uint32_t i = lane & 7u; i < n_in; i += 8) {
        const uint32_t key = start == kNotListed ? static_cast<uint32_t>(g_slots[static_cast<long long>(c) * kSlot + i])
                                                 : list[start + i] + (DT == 0 ? 0u : s_list_lo);
        f(c, acc, key);
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
      if ((lane & 7u) == 0 && c < n_local && !later) done(c, v, acc);
    }
    if (many) {
      __syncthreads();                           // (done writes cnt, by which the chunks are told apart)
      slot_keys_global<DT>(g_slots, cnt, n_local, [&](int c) { return (cnt[c] >> 16) && list_start[c] == kNotListed; }, f, done);
    }
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
  enum Leave { kDone = 0, kTimedOut = 1, kUnsound = 2 };
  const int left_as = [&]() -> int {
  // ---- the sample ----
  // A resident tensor: 1024 vectors of four elements, one per stratum, the same for
  // every CTA (each starts elsewhere in it, so that they do not all ask for the same lines at the
  // same time).  The margin is 3.5 standard deviations (a miss costs another pass over shared memory): at most 6 % of
  // the elements lie inside, for which the slots have twice the room.  Four times as many elements, with half the
  // bracket, cost 3 us more (up to 8 us of shared-memory atomics where many keys are equal) and saved 0.5.
  // A larger tensor, for which a miss is another read of it and a narrow bracket pays: every CTA
  // samples the whole tensor at places of its own (stratum G i + p of the G i-th row, p scrambled from
  // row to row so that no period of the data falls to one CTA) and reports where the threshold lies in
  // its own 4 thousand elements.  The CTAs' answers are independent draws whose median is the
  // threshold, however the elements are distributed, so the ones 2.5 sqrt(G) places (5 standard
  // deviations) to either side of the middle bound it: 0.4 % of the elements to each side, as the sum of
  // all histograms would give.  One exchange of one word per CTA, 4 us less than a window from CTA 0's part
  // and added-up histograms took.
  uint32_t lo = 1, hi = kKeyMax;
  constexpr int kPer = RES || DT == 0 ? 2 : 1;   // vectors per thread
  constexpr int kVecElems = RES ? 4 : EPV;       // elements of one
  constexpr int kVecWords = kVecElems * static_cast<int>(sizeof(E)) / 4;
  constexpr int kBinShift = Elem<DT>::kKeyBits - kSampleBinsLog2;
  constexpr int kFineShift = kBinShift > kSelBinsLog2 ? kBinShift - kSelBinsLog2 : 0;     // (!RES)
  uint4 v[kPer];
  {
    constexpr uint32_t kStrata = kPer * kThreads / (!RES && DT == 0 ? 2 : 1);     // of this CTA
    const uint32_t strata = RES ? kStrata : kStrata * G;
    const uint32_t n_vec = static_cast<uint32_t>(a.n / kVecElems);
    const float stride = static_cast<float>(n_vec) / static_cast<float>(strata);
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      uint32_t loc = u * kThreads + tid, part = 0;
      if (!RES && DT == 0) { part = loc & 1u; loc >>= 1; }         // two lanes share a stratum: 32 bytes
      if (RES) {
        loc = (loc + blockIdx.x * 37u) % kStrata;
      } else {
        const uint32_t at_row = blockIdx.x + __umulhi(hash_u32(loc + 0x9E3779B9u), static_cast<uint32_t>(G));
        loc = loc * G + (at_row >= static_cast<uint32_t>(G) ? at_row - G : at_row);
      }
      const float at = (static_cast<float>(loc) + static_cast<float>(hash_u32(loc) >> 8) * (1.0f / 16777216.0f)) * stride;
      uint32_t pos = static_cast<uint32_t>(at);
      if (!RES && DT == 0) pos = (pos & ~1u) + part;
      v[u] = make_uint4(0, 0, 0, 0);
      if (n_vec) {
        pos = min(pos, n_vec - 1);
        if (kVecWords == 4) {
          v[u] = __ldg(reinterpret_cast<const uint4*>(a.x) + pos);
        } else {
          const uint2 half = __ldg(reinterpret_cast<const uint2*>(a.x) + pos);
          v[u].x = half.x;
          v[u].y = half.y;
        }
      }
    }
  }

  // ---- set-up ----
  if (lane == 0) {                               // a warp's barriers are its own
    for (int s = 0; s < kSlotsPerWarp; ++s) tc::mbar_init(my_bars + 8 * s, 1);
    tc::fence_barrier_init();
  }
  __syncwarp();
  fly0 = start(false, 0);                        // (the others when the sample is there: it would queue behind them)
  if (tid == 0) {
    s_fail = 0;
    s_over = 0;
  }
  if (tid < 4) s_tot[tid] = 0;
  if (tid < key_room(G)) a.keys[blockIdx.x * key_room(G) + tid] = 0ull;      // (see the grid-wide exchange)
  for (int i = tid; i < kAuxBytes / 16; i += kThreads) reinterpret_cast<uint4*>(aux)[i] = make_uint4(0, 0, 0, 0);
  __syncthreads();

  unsigned long long execution = 0;
  if (master) {                                  // meanwhile CTA 0 prepares the exchanges
    if (tid == 0) {                              // (no value yet: what reads the store trusts the count)
      if (a.replayed) execution = atomicAdd(&g_executions, 1ull);
      a.hdr->status = SURGEON_OK;
      a.hdr->n_keep = 0;
    }
    // what a call of two rounds needs, the rest where a third is added
    prepare_exchanges(a, 1, spread ? kSelPhases : kFirstPhases, 0, spread ? kSelHists : kFirstRounds);
    if (!RES && tid < kSelPhases * kClaimSets) a.claims[tid * kClaimStride] = 0u;
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
    for (int e = 0; e < kVecElems; ++e) {
      const uint32_t key = ((DT == 0) ? w[e % 4] : (w[e >> 1] >> (16 * (e & 1)))) & kMask;
      const uint32_t bin = key >> kBinShift;
      if (key) atomicAdd(&hist[bin >> 1], 1u << (16 * (bin & 1)));   // (not the zeros, half of post-ReLU data)
    }
  }
  fly1 = start(false, 1);
  fly2 = start(false, 2);
  if (master && tid == 0) {                      // (by now its stores have arrived)
    s_tag = a.table_base + execution;
    fence_gpu();
    word_store(a.answer + (RES ? 0 : 1), a.token, execution);      // phase 0: (RES) prepared
  }
  // rank of the threshold inside the sample, and (RES) a margin of some standard deviations of a binomial count
  const float q = static_cast<float>(a.k) / static_cast<float>(a.n);
  constexpr float kOwn = static_cast<float>(kPer * kThreads * kVecElems);   // elements in this CTA's histogram
  const float up = q * kOwn, down = kOwn - up;   // of them above and below the threshold
  const bool no_hi = up < 16.0f, no_lo = down < 16.0f;     // (!RES) too few for a median that means something:
  uint32_t r_hi, r_lo = 0;                       // that side stays open, and the rank moves to the other
  if (RES) {
    const float delta = 3.5f * sqrtf(kOwn * q * (1.0f - q)) + 8.0f;
    r_hi = up - delta >= 1.0f ? static_cast<uint32_t>(up - delta) : 0u;                        // 0: none
    r_lo = up + delta <= kOwn - 1.0f ? static_cast<uint32_t>(up + delta) + 1u : 0u;            // 0: none
  } else {
    r_hi = static_cast<uint32_t>(no_hi ? up + sqrtf(up) + 2.0f : no_lo ? up - sqrtf(down) - 2.0f : up + 0.5f);
  }
  if (tid < 2) s_res[tid] = RES && tid == 0 && r_hi == 0 ? kSampleBins - 1u : 0u;
  if (tid < 2) s_res[4 + 2 * tid] = kThreads;    // (no thread has the rank)
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
#pragma unroll
    for (int which = 0; which < (RES ? 2 : 1); ++which) {
      // (a rank among the zeros lies below every counted bin: bin 0)
      const uint32_t want = which ? r_lo : r_hi;
      if (want && above < want && want <= above + sum) {
        s_res[4 + 2 * which] = tid;
        s_res[5 + 2 * which] = above;
      }
    }
    __syncthreads();
    if (warp < (RES ? 2 : 1) && s_res[4 + 2 * warp] < kThreads) {     // a warp for each rank, a lane per bin
      const uint32_t owner = s_res[4 + 2 * warp], want = warp ? r_lo : r_hi, bin = kSampleBins - 1u - 32u * owner - lane;
      const uint32_t c = (hist[bin >> 1] >> (16 * (bin & 1))) & 0xFFFFu;
      const uint32_t acc = s_res[5 + 2 * warp] + warp_excl_scan(c);
      if (acc < want && want <= acc + c) {
        s_res[warp] = bin;
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
      for (int e = 0; e < kVecElems; ++e) {
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
      if (!__syncthreads_and(ok)) return kTimedOut;
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
      if (tid == 0) {                            // (prepared behind a fence, above)
        word_store(a.answer, a.token, lo | (static_cast<unsigned long long>(hi) << 32));
      }
    } else {
      if (tid < 2) {
        ok = word_wait(a.answer + tid, a.token, &w);
        if (tid == 0) fence_gpu();
        s_ans[tid] = w;
      }
      if (!__syncthreads_and(ok)) return kTimedOut;
      if (tid == 0) s_tag = a.table_base + s_ans[1];
      lo = static_cast<uint32_t>(s_ans[0]);
      hi = static_cast<uint32_t>(s_ans[0] >> 32);
    }
  }

  // ---- the threshold ----
  // Every round counts the keys of [lo, hi] in bins of 2^shift keys, either in a pass over the chunks
  // (kRead) or from the keys that the last such pass listed (kRefine).
  uint32_t step = kRead, n_above = 0;            // n_above: keys above hi
  uint32_t first_lo = 1;                         // of the first round
  bool listed = false, loaded = true;            // (CTA 0) the last pass's lists are complete
  int shift = 0;
  int round = 0;
  uint32_t tau = 0, n_greater = 0;
  unsigned long long before = 0;
  for (;;) {
  for (; step <= kRefine; ++round) {
    if (round == kFirstRounds && tid == 1) fence_gpu();    // (it has read the answer) CTA 0 has cleared the other bins and answers
    const uint32_t range = hi - lo;
    shift = max(0, 32 - __clz(range) - kSelBinsLog2);
    __syncthreads();
    if (tid < kSelBins) hist[tid] = 0;
    if (tid < 4 && (step == kRead || tid == 1)) s_tot[tid] = 0;
    if (tid == 0 && step == kRead) {
      s_over = 0;
      s_list_n = 0;
      s_list_lo = lo;
    }
    __syncthreads();
    ulonglong2 prepared = make_ulonglong2(0, 0);   // (RES) CTA 0's first word, asked for ahead of its use
    if (RES && round == 0 && tid == 0) prepared = word_load(a.answer);
    uint32_t w_in = 0;                           // keys inside the bracket
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
        w_in += c_tot;
        if (c_tot > static_cast<uint32_t>(kSlot)) {
          // Massive ties.  If the chunk's keys inside the bracket all are one key, it is counted in
          // one go; if that holds everywhere with the same key, it is the threshold and the counts
          // are final without a list.
          const uint32_t k1 = one_key_of_chunk<DT>(region, cw[0], cw[WPL - 1], c_tot);
          if (lane == 0) s_over = 1;
          if (MODE == kStreamed && lane == 0) list_start[cl] = kNotListed;
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
          E* to = sl + warp_excl_scan(cc);
          take_set<DT, WPL, 2>(region, cw, [&](uint32_t i, E v) { to[i] = v & static_cast<E>(kMask); });
          __syncwarp();
          uint32_t at = kNotListed;
          if (MODE == kStreamed && (DT == 0 || range < 256u)) {
            if (lane == 0) at = atomicAdd(&s_list_n, c_tot);
            at = __shfl_sync(kFull, at, 0);
            if (at + c_tot > kListBytes / sizeof(L)) at = kNotListed;
          }
          if (MODE == kStreamed && lane == 0) list_start[cl] = static_cast<unsigned short>(at);
          for (uint32_t t = lane; t < c_tot; t += 32) {
            const uint32_t key = sl[t];
            atomicAdd(&hist[(key - lo) >> shift], 1u);
            kmax = max(kmax, key);
            kinv = max(kinv, ~key);
            if (!RES) {
              if (at != kNotListed) list[at + t] = static_cast<L>(DT == 0 ? key : key - lo);
              else g_slots[static_cast<long long>(cl) * kSlot + t] = static_cast<E>(key);
            }
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
        if (w_in) atomicAdd(&s_tot[1], w_in);
        if (kmax) atomicMax(&s_tot[2], kmax);
        if (kinv) atomicMax(&s_tot[3], kinv);
      }
    } else {
      auto add = [&](uint32_t key) {
        const uint32_t rel = key - lo;           // (below lo: wraps far above the range)
        if (rel <= range) {
          atomicAdd(&hist[rel >> shift], 1u);
          ++w_in;
        }
      };
      if (RES) {
        for (int c = warp; c < n_local; c += kWarps) slot_keys_warp<DT>(s_slots + c * kSlot, cnt[c] >> 16, add);
      } else if (spread) {
        slot_keys_global<DT>(g_slots, cnt, n_local, [](int) { return true; }, [&](int, uint32_t&, uint32_t key) { add(key); }, [](int, uint32_t, uint32_t) {});
      } else {
        listed_keys([&](int, uint32_t&, uint32_t key) { add(key); }, [](int, uint32_t, uint32_t) {});
      }
      w_in = warp_sum(w_in);
      if (lane == 0 && w_in) atomicAdd(&s_tot[1], w_in);
    }
    if (RES && round == 0 && tid == 0) {         // CTA 0 has zeroed the histograms
      if (prepared.x != a.token && !word_wait(a.answer, a.token, &prepared.y)) s_fail = 1;
      if (!master) s_tag = a.table_base + prepared.y;
      fence_gpu();
    }
    __syncthreads();
    if (s_fail) return kTimedOut;
    uint32_t* gh = a.hist + round * kSelBins;
    if (tid < kSelBins) {
      const uint32_t h = hist[tid];
      if (h) atomicAdd(&gh[tid], h);
    }
    if (tid == 0) {
      // reported: how many keys this CTA has put into the bins and the count above them, whether a list overflowed, and
      // the one key inside (0: none, ~0: several)
      const uint32_t n_up = step == kRead ? s_tot[0] : 0u;
      if (n_up) atomicAdd(above_count(a, round), n_up);
      const uint32_t one = s_tot[2] == 0u ? 0u : (s_tot[2] == ~s_tot[3] ? s_tot[2] : 0xFFFFFFFFu);
      if (spread) fence_gpu();                   // (the counts and lists, which other CTAs will read)
      word_store(a.arrive + phase * kSelMaxCtas + blockIdx.x, a.token,
                 (static_cast<unsigned long long>(one) << 32) | (n_up + s_tot[1]) | (s_over << 31));
    }
    // What the CTA has above and in each of the first bins (fp32, whose bins are no single keys: above and inside the bracket),
    // for the others: see the last exchange.  CTA 0 when it has answered.
    const bool shown = !spread && round == 0;
    auto show = [&]() {
      if (DT == 0) {
        if (tid == 0 && SURGEON_IN_BOUNDS(blockIdx.x, table_entries(a.n_chunks, DT), &a.hdr->status))
          word_store(a.table + blockIdx.x, s_tag, (static_cast<unsigned long long>(s_tot[0]) << 32) | s_tot[1]);
      } else {
        uint32_t all;
        const uint32_t mine = my_bin(hist), bin = kSelBins - 1u - tid, up = count_above_mine(mine, s_warp, &all) + s_tot[0];
        if (tid < kSelBins && bin < static_cast<uint32_t>(table_bins(DT)) && bin <= range >> shift &&
            SURGEON_IN_BOUNDS(blockIdx.x * table_bins(DT) + bin, table_entries(a.n_chunks, DT), &a.hdr->status))
          word_store(a.table + blockIdx.x * table_bins(DT) + bin, s_tag, (static_cast<unsigned long long>(up) << 32) | mine);
      }
    };
    if (shown) { first_lo = lo; if (!master) show(); }
    if (master) {
      unsigned long long v = 0;
      int ok = 1;
      if (tid < G) {
        ok = word_wait(a.arrive + phase * kSelMaxCtas + tid, a.token, &v, a.stall != 0);
        if (spread) fence_gpu();
        a.arrive[phase * kSelMaxCtas + tid].x = 0ull;
      }
      if (!__syncthreads_and(ok)) return kTimedOut;
      const uint32_t one = static_cast<uint32_t>(v >> 32);
      const uint32_t w_max = __reduce_max_sync(kFull, one), w_inv = __reduce_max_sync(kFull, one ? ~one : 0u);
      const uint32_t w_over = __any_sync(kFull, (static_cast<uint32_t>(v) >> 31) != 0u) ? 1u : 0u;
      const uint32_t w_sum = __reduce_add_sync(kFull, static_cast<uint32_t>(v) & 0x7FFFFFFFu);
      __shared__ uint4 s_red[kWarps];
      __shared__ uint32_t s_up;
      if (lane == 0) s_red[warp] = make_uint4(w_sum, w_max, w_inv, w_over);
      uint32_t b, n_in, above, n_up, all = 0;
      for (uint32_t spins = 0;; ++spins) {       // until everything that was reported has arrived in the bins
        b = tid < kSelBins ? count_load(gh + kSelBins - 1 - tid) : 0u;
        if (tid == 0) s_up = count_load(above_count(a, round));
        above = count_above_mine(b, s_warp, &n_in);
        n_up = s_up;
        if (spins == 0) all = __reduce_add_sync(kFull, lane < kWarps ? s_red[lane].x : 0u);
        if (n_in + n_up == all || spins > (1u << 18)) break;
        __syncthreads();
      }
      if (n_in + n_up != all) return kTimedOut;
      const uint4 red = lane < kWarps ? s_red[lane] : make_uint4(0, 0, 0, 0);
      const uint32_t key_max = __reduce_max_sync(kFull, red.y);
      const uint32_t key_inv = __reduce_max_sync(kFull, red.z);
      const bool over = __any_sync(kFull, red.w != 0u);
      const bool was_read = step == kRead;
      if (was_read) { n_above = n_up; listed = !over; }
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
        else step = s_res[2] <= kKeysAtOnce && shift <= 2 * kSelBinsLog2 ? kKeys : kRefine;
      }
      if (step <= kRefine && !spread && round + 1 == kFirstRounds) {         // an unusual call: prepare the rest
        prepare_exchanges(a, kFirstPhases, kSelPhases, kFirstRounds, kSelHists);
        __syncthreads();
        if (tid == 0) fence_gpu();
      }
      if (tid == 0) {
        if (spread) fence_gpu();
        word_store(a.answer + phase * (kSelMaxCtas + 2), a.token, lo | (static_cast<unsigned long long>(hi) << 32));
        word_store(a.answer + phase * (kSelMaxCtas + 2) + 1, a.token, n_above | (static_cast<unsigned long long>(step) << 32));
        if (phase == 1) a.answer[0].x = a.answer[1].x = 0ull;
      }
      if (!spread && step == kKeys && G > 1 && tid < G) fence_gpu();       // the key words of all CTAs have been cleared
      if (shown && step != kKeys) {              // (else nobody looks)
        __syncthreads();
        show();
      }
    } else {
      if (tid < 2) {
        unsigned long long v = 0;
        if (!word_wait(a.answer + phase * (kSelMaxCtas + 2) + tid, a.token, &v, a.stall != 0)) s_fail = 1;
        if (spread) fence_gpu();                 // the counts and lists of the other CTAs
        s_ans[tid] = v;
      }
      __syncthreads();
      if (s_fail) return kTimedOut;
      lo = static_cast<uint32_t>(s_ans[0]);
      hi = static_cast<uint32_t>(s_ans[0] >> 32);
      n_above = static_cast<uint32_t>(s_ans[1]);
      step = static_cast<uint32_t>(s_ans[1] >> 32);
    }
    ++phase;
    if (round + 1 >= kSelHists && step <= kRefine) {   // cannot happen: a miss, three levels and a pass for ties are the most
      if (tid == 0) atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_INTERNAL));
      return kUnsound;
    }
  }

  // ---- what this CTA has above the threshold (or above its bin) and at it ----
  if (step == kRecount) {                        // the lists overflowed: count once more from the chunks
    __syncthreads();
    auto recount = [&](int c, unsigned char* region) -> bool {
      const uint32_t both = count_chunk<DT>(region, lo);
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
    if (spread && !meet()) return kTimedOut;
  }
  // The threshold is known after one round: no last exchange.  The CTAs have shown what they have above each bin and in it, so
  // every one adds up what lies before it, and all, for itself.
  const uint32_t known_bin = DT == 0 || step == kZero ? 0u : (lo - first_lo) >> shift;
  const bool direct = !spread && round == 1 && (step == kZero || step == kOneKey || (DT != 0 && step != kKeys)) && known_bin < static_cast<uint32_t>(table_bins(DT));
  ulonglong2 entry = make_ulonglong2(0, 0);      // asked for ahead of its use
  if (direct && tid < G) entry = word_load(a.table + tid * table_bins(DT) + known_bin);
  if (tid == 0) s_nkeys = 0;
  __syncthreads();
  if (s_fail) return kTimedOut;
  uint32_t n_gt = 0, n_eq = 0;
  if (step == kListed || step == kKeys) {
    // acc: keys above hi, and (upper half) keys of [lo, hi]
    auto report = [&](int c, uint32_t& acc, uint32_t key) {
      if (key > hi) ++acc;
      else if (key >= lo) {
        acc += 0x10000u;
        if (step == kKeys) {
          const uint32_t at = atomicAdd(&s_nkeys, 1u);
          if (at < static_cast<uint32_t>(key_room(G))) {
            key_store(a.keys + blockIdx.x * key_room(G) + at, key_tag(a.token, phase), key);
            s_bin_key[at] = key;
            s_bin_chunk[at] = c;
          }
        }
      }
    };
    auto done = [&](int c, uint32_t v, uint32_t acc) {       // (one lane)
      acc += v & 0xFFFFu;
      if (step == kListed) cnt[c] = acc;
      else if (MODE == kStreamed) list_acc[c] = static_cast<unsigned short>(acc);
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
    } else if (spread) {
      slot_keys_global<DT>(g_slots, cnt, n_local, [](int) { return true; }, report, done);
    } else {
      listed_keys(report, done);
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
  if (direct) {
    tau = lo; n_greater = n_above;
    unsigned long long v = 0;
    int ok = 1;
    if (tid < G) {
      const unsigned long long tag = s_tag;
      v = entry.y;
      if (entry.x != tag) ok = word_wait(a.table + tid * table_bins(DT) + known_bin, tag, &v);
      if (step == kZero) {                       // what is neither above the first bin nor in the bins is a tie
        const uint32_t gt = static_cast<uint32_t>(v >> 32) + static_cast<uint32_t>(v);
        const long long from = static_cast<long long>(a.n_chunks) * tid / G * (32 * EPR);
        const long long to = min(a.n, static_cast<long long>(a.n_chunks) * (tid + 1) / G * (32 * EPR));
        v = (static_cast<unsigned long long>(gt) << 32) | static_cast<uint32_t>(to - from - gt);
      }
    }
    if (!__syncthreads_and(ok)) return kTimedOut;
    unsigned long long sum = v, first = tid < static_cast<int>(blockIdx.x) ? v : 0ull;     // of all CTAs, of those before this one
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      sum += __shfl_xor_sync(kFull, sum, o);
      first += __shfl_xor_sync(kFull, first, o);
    }
    __shared__ unsigned long long s_first[kWarps];
    if (lane == 0) { s_warp64[warp] = sum; s_first[warp] = first; }
    __syncthreads();
    sum = lane < kWarps ? s_warp64[lane] : 0ull;
    first = lane < kWarps ? s_first[lane] : 0ull;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      sum += __shfl_xor_sync(kFull, sum, o);
      first += __shfl_xor_sync(kFull, first, o);
    }
    before = __shfl_sync(kFull, first, 0);
    sum = __shfl_sync(kFull, sum, 0);
    const bool none = a.drop_zeros && tau == 0u;
    const long long quota = none ? 0 : static_cast<long long>(a.k) - n_greater, eq_all = static_cast<long long>(sum & 0xFFFFFFFFull);
    const long long n_stored = none ? static_cast<long long>(n_greater) : static_cast<long long>(a.k);
    // (as at the exchange: nothing is stored if the counts do not add up; all CTAs see the same)
    if (static_cast<long long>(sum >> 32) != n_greater || quota < 0 || n_greater + (eq_all < quota ? eq_all : quota) != n_stored) {
      if (master && tid == 0) atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_INTERNAL));
      return kUnsound;
    }
    if (master && tid == 0) {
      a.hdr->threshold_key = tau;
      a.hdr->n_keep = n_stored;
      a.hdr->n_greater = n_greater;
      a.hdr->tie_quota = quota;
      a.offsets[(a.n + SURGEON_BLOCK - 1) >> kBlockShift] = static_cast<uint32_t>(n_stored);   // the sentinel entry
    }
    break;
  }
  n_gt = warp_sum(n_gt);
  n_eq = warp_sum(n_eq);
  if (lane == 0) s_warp64[warp] = (static_cast<unsigned long long>(n_gt) << 32) | n_eq;
  __syncthreads();
  if (tid == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < kWarps; ++w) t += s_warp64[w];
    word_store(a.arrive + phase * kSelMaxCtas + blockIdx.x, a.token, t);
  }

  // ---- last exchange: the threshold, and every CTA's place ----
  tau = lo; n_greater = n_above;
  bool again = false;                            // a CTA has more keys than it can report: narrow the bin first
  if (master) {
    // two threads per CTA, which share its keys
    const int who = tid >> 1;
    unsigned long long v = 0;
    int ok = 1;
    if (who < G) {
      ok = word_wait(a.arrive + phase * kSelMaxCtas + who, a.token, &v);
      if (!(tid & 1)) a.arrive[phase * kSelMaxCtas + who].x = 0ull;
    }
    if (step == kKeys) {
      const uint32_t n_k = static_cast<uint32_t>(v);
      const bool fits = n_k <= static_cast<uint32_t>(key_room(G));
      const unsigned long long* mine = a.keys + who * key_room(G) + (tid & 1);
      // the keys, with their CTA, in shared memory; their histogram by the upper bits of key - lo
      uint32_t* got = hist + kSelBins;           // [kKeysAtOnce]
      uint32_t* nk = got + kKeysAtOnce;          // [kSelMaxCtas] keys of a CTA above the threshold, and (upper half) ties
      unsigned char* owner = reinterpret_cast<unsigned char*>(nk + kSelMaxCtas);
      const int coarse = shift > kSelBinsLog2 ? shift - kSelBinsLog2 : 0;
      if (tid < kSelBins) hist[tid] = 0;
      if (tid < kSelMaxCtas) nk[tid] = 0;
      if (tid == 0) s_res[6] = s_res[7] = 0;
      __syncthreads();
      const int turns = __reduce_max_sync(kFull, fits ? static_cast<int>((n_k + 7u) / 8u) : 0);
#pragma unroll 1
      for (int turn = 0; turn < turns; ++turn) { // four keys of each thread at a time
        unsigned long long w[4];
        bool late;
        uint32_t spins = 0;
        const uint32_t first = 8u * turn + (tid & 1u), left = fits && n_k > first ? n_k - first : 0u;      // word u: 2 u < left
        do {
          late = false;
#pragma unroll
          for (int u = 0; u < 4; ++u) w[u] = key_load_if(mine + 8 * turn + 2 * u, 2u * u < left, key_tag(a.token, phase), lo);
#pragma unroll
          for (int u = 0; u < 4; ++u)            // (a number outside the bin is no index below)
            late |= static_cast<uint32_t>(w[u] >> 32) != key_tag(a.token, phase) || static_cast<uint32_t>(w[u]) - lo > hi - lo;
        } while (late && ++spins < (1u << 20));
        if (late) ok = 0;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t key = static_cast<uint32_t>(w[u]);
          const bool got_one = !late && 2u * u < left;
          const uint32_t have = __ballot_sync(kFull, got_one);
          uint32_t at = 0;
          if (lane == 0 && have) at = atomicAdd(&s_res[6], __popc(have));
          at = __shfl_sync(kFull, at, 0) + __popc(have & lanemask_lt());
          if (got_one && at < kKeysAtOnce) {
            got[at] = key;
            owner[at] = static_cast<unsigned char>(who);
            atomicAdd(&hist[(key - lo) >> coarse], 1u);
          }
        }
      }
      again = __syncthreads_or(!fits) != 0;
      if (!__syncthreads_and(ok)) return kTimedOut;
      if (!again) {
        const uint32_t n_got = min(s_res[6], kKeysAtOnce);
        uint32_t all;
        uint32_t b = my_bin(hist);
        place_rank(b, count_above_mine(b, s_warp, &all), a.k - n_above, s_res);
        __syncthreads();
        const uint32_t in_bin = s_res[2], bin = lo + (s_res[0] << coarse);
        tau = bin;
        n_greater = n_above + s_res[1];
        if (coarse) {                            // its keys, which a warp can hold (few lie in a bin of 512)
          __shared__ uint32_t s_few[32];
          if (in_bin > 32u) hist[tid] = 0;       // (massive ties: their low bits are counted)
          __syncthreads();
#pragma unroll 1
          for (uint32_t i = tid; i < n_got; i += kThreads) {
            const uint32_t rel = got[i] - bin;   // (below the bin: wraps)
            if (rel >> coarse == 0u) {
              if (in_bin <= 32u) s_few[atomicAdd(&s_res[7], 1u)] = got[i];
              else atomicAdd(&hist[rel], 1u);
            }
          }
          __syncthreads();
          if (in_bin <= 32u) {                   // every warp ranks them
            const uint32_t k0 = lane < in_bin ? s_few[lane] : 0u;
            uint32_t larger = 0;
#pragma unroll 1
            for (uint32_t i = 0; i < in_bin; ++i) larger += __shfl_sync(kFull, k0, i) > k0 ? 1u : 0u;
            // the threshold: the smallest key with fewer than the wanted rank above it
            tau = __reduce_min_sync(kFull, lane < in_bin && larger < a.k - n_greater ? k0 : 0xFFFFFFFFu);
            n_greater += __popc(__ballot_sync(kFull, lane < in_bin && k0 > tau));
          } else {
            b = my_bin(hist);
            place_rank(b, count_above_mine(b, s_warp, &all), a.k - n_greater, s_res + 3);
            __syncthreads();
            tau += s_res[3];
            n_greater += s_res[4];
          }
        }
#pragma unroll 1
        for (uint32_t i = tid; i < n_got; i += kThreads)
          if (got[i] >= tau) atomicAdd(&nk[owner[i]], got[i] > tau ? 1u : 0x10000u);
        __syncthreads();
        if (who < G) v = (((v >> 32) + (nk[who] & 0xFFFFu)) << 32) | (nk[who] >> 16);
      }
    } else if (!__syncthreads_and(ok)) {
      return kTimedOut;
    }
    // exclusive scan over the CTAs
    if (tid & 1) v = 0;
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
    if (again && !spread && round == kFirstRounds) {         // an unusual call: prepare what its next rounds need
      prepare_exchanges(a, kFirstPhases, kSelPhases, kFirstRounds, kSelHists);
      __syncthreads();
      if (tid == 0) fence_gpu();
      __syncthreads();
    }
    if (who < G && !(tid & 1)) word_store(a.answer + phase * (kSelMaxCtas + 2) + 2 + who, a.token, base + incl - v);
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
    if (verdict == 2u) return kUnsound;
  } else {
    __shared__ unsigned long long s_last[3];
    if (tid < 3) {
      unsigned long long v = 0;
      const int which = tid < 2 ? tid : 2 + static_cast<int>(blockIdx.x);
      if (!word_wait(a.answer + phase * (kSelMaxCtas + 2) + which, a.token, &v)) s_fail = 1;
      s_last[tid] = v;
    }
    __syncthreads();
    if (s_fail) return kTimedOut;
    if (s_last[1] == 2ull) return kUnsound;
    again = s_last[1] == 1ull;
    tau = static_cast<uint32_t>(s_last[0]);
    n_greater = static_cast<uint32_t>(s_last[0] >> 32);
    before = s_last[2];
  }
  ++phase;
  // They have been read.  (Not needed: they carry this phase's tag.  Without a place where the paths of all steps meet, small
  // calls that report no keys took 2-4 us longer.)
  if (step == kKeys && tid < min(static_cast<int>(s_nkeys), key_room(G))) a.keys[blockIdx.x * key_room(G) + tid] = 0ull;
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
      uint32_t both = MODE == kStreamed ? list_acc[c] : static_cast<uint32_t>(prefix[c]);
#pragma unroll 1
      for (int i = 0; i < n_bin; ++i)
        if (s_bin_chunk[i] == c && s_bin_key[i] >= tau) both += s_bin_key[i] > tau ? 1u : 0x10000u;
      cnt[c] = both;
    }
    __syncthreads();
  }
  if (RES) {                                     // every warp for itself: at most 48 chunks
    uint32_t up[2], tie[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = 32 * j + static_cast<int>(lane);
      const uint32_t v = c < n_local ? cnt[c] : 0u;
      up[j] = v & 0xFFFFu;
      tie[j] = v >> 16;
    }
    unsigned long long base = before;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = 32 * j + static_cast<int>(lane);
      const uint32_t u0 = warp_excl_scan(up[j]), t0 = warp_excl_scan(tie[j]);
      if (c < n_local && c % kWarps == warp) prefix[c] = base + ((static_cast<unsigned long long>(u0) << 32) | t0);
      base += (static_cast<unsigned long long>(__shfl_sync(kFull, u0 + up[j], 31)) << 32) | __shfl_sync(kFull, t0 + tie[j], 31);
    }
    __syncwarp();
  } else {
  unsigned long long carry = before;
  constexpr int kScan = 4;                       // consecutive chunks per thread
#pragma unroll 1
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

  }
  // ---- emit ----
  if (RES) {
    run_resident(false, [&](int c, unsigned char* region) -> bool {
      return emit_chunk<DT>(a, region, c, tau, quota, prefix[c - c_begin], cnt[c - c_begin] >> 16, n_stored);
    });
    return kDone;
  }
  // From the end, where the ring (not claimed: its places still hold the last three) and the L2 cache have it.
  unsigned long long at_next = 0;                // (claimed) place and ties of the next chunk, fetched one chunk ahead
  uint32_t n_next = 0;
  if (spread) {
    if (!meet()) return kTimedOut;               // every CTA's places are known to all
    tc::fence_proxy_async();
    __syncwarp();
    begin_pass(true);
    if (fly0 < a.n_chunks) { at_next = prefix[fly0 - c_begin]; n_next = cnt[fly0 - c_begin]; }
  }
  int i = n_mine - 1;                            // (not claimed) the next one
  int s = spread || i < 0 ? 0 : i % kSlotsPerWarp;
#pragma unroll 1
  while (spread ? fly0 < a.n_chunks : i >= 0) {
    const int c = spread ? fly0 : chunk_of(i);
    if ((spread || i + kSlotsPerWarp < n_mine) && !arrived(c, s)) {
      atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
      break;
    }
    unsigned long long at = at_next;
    uint32_t n_at = n_next;
    if (!spread) { at = prefix[c - c_begin]; n_at = cnt[c - c_begin]; }
    else if (fly1 < a.n_chunks) { at_next = prefix[fly1 - c_begin]; n_next = cnt[fly1 - c_begin]; }
    const bool written = emit_chunk<DT>(a, my_ring + s * kChunkBytes, c, tau, quota, at, n_at >> 16, n_stored);
    int c_load;                                  // what the place takes next
    if (spread) {
      fly0 = fly1; fly1 = fly2;
      c_load = next();
      fly2 = c_load;
      if (c_load < a.n_chunks) fly2 = c_load = a.n_chunks - 1 - c_load;
    } else {
      c_load = i >= kSlotsPerWarp ? chunk_of(i - kSlotsPerWarp) : a.n_chunks;
      --i;
    }
    if (c_load < a.n_chunks) {
      if (written) tc::fence_proxy_async();      // this warp's writes to the place precede the next TMA fill
      __syncwarp();                              // every lane has read the place
      issue(c_load, s);
    }
    s = spread ? (s == 2 ? 0 : s + 1) : (s == 0 ? 2 : s - 1);
  }
  return kDone;
  }();

  // A wait gave up somewhere: the loads under way are waited for (with a limit) as well, and the CTA takes back what it
  // has stored for the others: a replay of a captured call carries the same token and must not find it.
#pragma unroll 1
  for (int s = 0; s < kSlotsPerWarp; ++s)
    if ((under_way >> s) & 1u) landed(s);
  if (left_as == kTimedOut) {
    if (tid == 0) atomicMax(&a.hdr->status, static_cast<uint32_t>(SURGEON_ERR_TIMEOUT));
    if (tid < kSelPhases) a.arrive[tid * kSelMaxCtas + blockIdx.x].x = 0ull;
    if (master)
      for (int i = tid; i < kSelPhases * (kSelMaxCtas + 2); i += kThreads) a.answer[i].x = 0ull;
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
// Algorithm 1, Reshape step: one warp rebuilds 1024 elements (32 bitmap words) of the dense tensor at a time.
// The piece's packed values are one contiguous run: they are staged in shared memory with 16-byte
// asynchronous copies; a lane then puts the values of its bitmap word (a loop over the set bits, about 8
// instructions per kept element of the fullest word) into its row of a zeroed tile, and the tile
// leaves as 16-byte vectors.  Bound by the memory: a warp keeps the values of its next piece and the words of the one
// after that in flight.
// bf16, 77 MB, 30 % kept: 43.0 -> 34.8 us; fp32, 131 MB, 40 % kept: 90 -> 69; 1.1 GB, 70 % kept: 785 -> 572 (4.0 TB/s).
constexpr int kDecWarps = 8;
constexpr int kDecElems = 1024;
template <int DT>
__host__ __device__ constexpr int dec_stage_bytes() {                // values of a piece, with alignment slack
  return kDecElems * static_cast<int>(sizeof(typename Elem<DT>::type)) + 16;
}
template <int DT>
__host__ __device__ constexpr int dec_warp_bytes() {                 // the tile, and the values of two pieces
  return kDecElems * static_cast<int>(sizeof(typename Elem<DT>::type)) + 2 * dec_stage_bytes<DT>();
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
  unsigned char* stages = tile + kDecElems * sizeof(E);
  const uint32_t lane = lane_id();
  // vectors of a row are XORed with the row's number: lanes at the same place of their rows differ in banks
  auto swz = [](uint32_t row) { return DT == 0 ? (row & 7u) : ((row >> 1) & 3u); };
  const long long n_chunks = (n + kDecElems - 1) / kDecElems;
  const long long n_words = (n + 31) / 32;
  const long long n_blocks = (n + SURGEON_BLOCK - 1) >> kBlockShift;
  const long long warps = (static_cast<long long>(gridDim.x) * blockDim.x) >> 5;
  const uint32_t n_vals = offsets[n_blocks];
  struct Piece { uint32_t word, first; };        // this lane's word; the packed place of the piece's first value
  auto fetch = [&](long long chunk) {
    Piece q{0u, 0u};
    if (chunk < n_chunks) {
      const long long w_idx = chunk * 32 + lane;
      if (w_idx < n_words) q.word = __ldg(bitmap + w_idx);
      q.first = __ldg(offsets + chunk * (kDecElems / SURGEON_BLOCK));
    }
    return q;
  };
  auto copy_values = [&](const Piece& q, unsigned char* stage) {     // from the vector that holds the first one on
    const uint32_t total = __reduce_add_sync(kFull, __popc(q.word));
    const uint32_t a0 = q.first & ~static_cast<uint32_t>(EPV - 1);
    const uint32_t n_vec = total ? (q.first + total - a0 + EPV - 1) / EPV : 0u;
#pragma unroll 1
    for (uint32_t v = lane; v < n_vec; v += 32) {
      const uint32_t e0 = a0 + v * EPV;
      if (e0 + EPV <= n_vals) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(stage + v * 16)), "l"(values + e0) : "memory");
      } else {                                   // the vector that ends past the last value
        E* to = reinterpret_cast<E*>(stage) + v * EPV;
        for (uint32_t e = 0; e < static_cast<uint32_t>(EPV) && e0 + e < n_vals; ++e) to[e] = values[e0 + e];
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  long long chunk = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  Piece now = fetch(chunk), next = fetch(chunk + warps);
  uint32_t which = 0;
  copy_values(now, stages);
#pragma unroll 1
  for (; chunk < n_chunks; chunk += warps, which ^= 1u) {
    const Piece after = fetch(chunk + 2 * warps);
    copy_values(next, stages + (which ^ 1u) * dec_stage_bytes<DT>());
    unsigned char* row = tile + lane * (32 * sizeof(E));
#pragma unroll
    for (int j = 0; j < kRowVecs; ++j) reinterpret_cast<uint4*>(row)[j] = make_uint4(0, 0, 0, 0);
    uint32_t word = now.word;
    const uint32_t excl = warp_excl_scan(__popc(word));
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    const E* src = reinterpret_cast<const E*>(stages + which * dec_stage_bytes<DT>()) + (now.first & (EPV - 1)) + excl;
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
    now = next;
    next = after;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
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

unsigned long long random_number() {
  std::random_device rd;
  const unsigned long long t = static_cast<unsigned long long>(
      std::chrono::steady_clock::now().time_since_epoch().count());
  return ((static_cast<unsigned long long>(rd()) << 32) | rd()) ^ (t << 20);
}
// A value that no other call of this or another process carries (see the grid-wide exchange).
unsigned long long next_token() {
  static std::atomic<unsigned long long> counter{random_number()};
  return counter.fetch_add(1, std::memory_order_relaxed);
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
  static const unsigned long long table_base = random_number();
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess) {        // (not known: counted; the launch will say what is wrong)
    capture = cudaStreamCaptureStatusActive;
    cudaGetLastError();
  }
  a.replayed = capture != cudaStreamCaptureStatusNone;
  a.table_base = a.replayed ? table_base : ~a.token;
  a.hdr = out.header; a.bitmap = out.bitmap; a.values = out.values; a.offsets = out.block_offsets;
  a.arrive = reinterpret_cast<ulonglong2*>(ws + L.arrive);
  a.answer = reinterpret_cast<ulonglong2*>(ws + L.answer);
  a.keys = reinterpret_cast<unsigned long long*>(ws + L.keys);
  a.hist = reinterpret_cast<uint32_t*>(ws + L.hist);
  a.claims = reinterpret_cast<uint32_t*>(ws + L.claims);
  a.cnt = reinterpret_cast<uint32_t*>(ws + L.cnt);
  a.prefix = reinterpret_cast<unsigned long long*>(ws + L.prefix);
  a.table = reinterpret_cast<ulonglong2*>(ws + L.table);
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
  // of the GPU only where the counts do not fit (on a quarter, 134 MB fp32, claimed and streamed: 40 % kept 249 and 233 us,
  // 5 % kept 216 and 199, 70 % kept 250 and 252)
  const bool claimed = a.n_chunks > grid * (share ? kMaxLocalChunks : 512);
  const bool resident = (a.n_chunks + grid - 1) / grid <= kResidentChunks;
  const void* kernel = resident  ? reinterpret_cast<const void*>(prune_kernel<DT, kResident>)
                       : claimed ? reinterpret_cast<const void*>(prune_kernel<DT, kClaimed>)
                                 : reinterpret_cast<const void*>(prune_kernel<DT, kStreamed>);
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
  // the CTAs that a device holds: two per SM in fp32, four in bf16
  const long long cap = (act.dt == 0 ? 2LL : 4LL) * sm_count();
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
