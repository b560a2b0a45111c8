// Fragment scan (paper Section 5): every 64-byte window of a disk image that starts at a
// multiple of 4 bytes is looked up among the whole 64-byte fragments of the master files, to
// find small files (logos, small images) embedded in other files at any 32-bit offset.
//
// Work layout. A tile is one warp's work: 32 x WPT consecutive windows. Each warp stages its own
// tiles (the window starts plus the last window's 60-byte tail) into its own shared-memory
// buffer with 1-D bulk TMA copies issued by its lane 0, completion on the warp's own mbarrier,
// every wait bounded; warps of a block never wait for one another, so a warp that meets a
// candidate (an L2 probe) holds up no one. Lane l takes windows [WPT l, WPT l + WPT) of the tile;
// with WPT odd the 32 lanes read 32 different banks at every step.
//
//   djb2-64 (Eq. 1) is rolled. With P(x) the base-33 Horner value of a 4-byte word x and
//   g = h - 5381 * 33^64, a window W_k of words x_k .. x_{k+15} has g(W_k) = sum_q
//   P(x_{k+q}) 33^{4 (15 - q)}, so g(W_{k+1}) = 33^4 g(W_k) - 33^64 P(x_k) + P(x_{k+16})
//   (mod 2^64): after a lane's first window each one costs one word and a few multiply-adds.
//   The same recurrence holds mod 2^32, so the count kernel rolls only the low word of h: two
//   multiply-adds a window. Its filters are functions of that word (but see frag_key_class): two bits
//   of one word of a 2^20-bit filter in shared memory (loaded once per block), then, for the windows
//   that pass, one word of a Bloom filter in global memory. What is left computes its whole h and is looked up.
//   MD5 is computed per window (two compressions, or one without the padding block); there the
//   hash dominates and the global Bloom word is tested directly.
//
// Passes, over the tiles of all images of a call. The count kernel hashes every window, filters it,
// resolves the candidates (probe; byte confirmation for djb2), writes each tile's triple count and, for
// a tile with triples, an entry of the hit list: which windows of each lane have any. An exclusive scan gives every tile
// its output offset; the emit kernel looks the listed windows up again and writes their triples
// in window order. (Hit records instead of lookups done twice would need room for every window.)
// The lists' masks take 128 bytes per tile, 4.3% of the image for djb2 and 3.2% for MD5, and at
// most 512 MiB; a listed tile beyond that has all its windows looked up again.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <type_traits>

#include "cv_launch.h"
#include "scan_kernel.cuh"

namespace cvk {

// Tile geometry per signature (a tile is one warp's work).
template <int SIG>
struct FragGeom {
  static constexpr bool kRolled = SIG == kSigDjb2;
  // 32 warps per SM. The rolled kernel's blocks stay and share one copy of the filter; an MD5 warp
  // hashes one tile (some 70 us) and a block of two such warps ends, so that the hardware deals the
  // blocks out: with a fixed share of the tiles per warp the same kernel took 1,660 against 1,506 us
  // (256 MiB), because the scheduler favours some warps of an SM. Tiles with repeated windows are
  // done earlier: blocks of four warps 1,231 us, of two 1,227, of one (of 29 windows a lane, for the
  // blocks' shared memory) 1,244.
  static constexpr int kThreads = kRolled ? 1024 : 64;   // block size
  static constexpr int kMinBlocks = kRolled ? 1 : 16;     // resident blocks per SM
  static constexpr int kWarps = kThreads / 32;
  static constexpr int kWPT = kRolled ? 23 : 31;  // windows per lane per tile (odd)
  // Rolled: windows per lane that can wait for the second filter. They wait in the lane's part of
  // the tile, from its word 15 on, where the words are read by this lane alone, each before the
  // entry that takes its place is written.
  static constexpr int kQueue = kWPT - 15;
  static constexpr uint32_t kTileWin = 32 * kWPT;
  static constexpr uint32_t kTileStep = kTileWin * kFragStride;  // bytes between tile starts
  static constexpr uint32_t kTileBytes = kTileStep + 64;         // bytes staged per tile
  static constexpr bool kL1 = kRolled;                           // shared-memory filter
  static constexpr uint32_t kL1Off = kWarps * kTileBytes;  // filter after the warps' buffers
  // not rolled: per warp the windows to be hashed (16-bit numbers) and the lanes' candidate masks
  static constexpr uint32_t kListBytes = kRolled ? 0 : kTileWin * 2 + 128;
  static constexpr uint32_t kSmemCount = kL1Off + (kL1 ? kFragL1Bytes : 0) + kWarps * kListBytes;
  static_assert(kWPT % 2 == 1 && kWPT <= 32 && (!kRolled || kQueue > 0), "odd window count, masks of 32 bits");
  static_assert(kTileBytes % 16 == 0 && kTileStep % 16 == 0, "bulk copies of whole 16-byte chunks");
  static_assert(kSmemCount <= 227 * 1024, "shared memory of one block");
};

__host__ __device__ constexpr uint64_t pow33(int e) {
  uint64_t r = 1;
  for (int i = 0; i < e; i++) r *= 33u;
  return r;
}
constexpr uint64_t kD33x4 = pow33(4);
constexpr uint64_t kD33x64 = pow33(64);
constexpr uint64_t kDjbInit = 5381ull * pow33(64);  // 5381 * 33^64: the initial value's share

struct FragParams {
  TableView tab;
  FragImages images;             // their tiles are numbered through
  uint64_t n_tiles;              // of all images
  uint64_t* tile_ntrip;          // count: triples per tile
  const uint64_t* tile_off;      // emit: output offset per tile
  uint32_t* hit_tiles;           // the tiles with triples, in any order
  uint32_t* hit_masks;           // per listed tile and lane: its windows with triples
  uint32_t* n_hit_tiles;         // their number (device), zero before the count
  uint32_t mask_cap;             // listed tiles that have masks
  const uint64_t* total;         // emit: the triples of all images
  MatchOut* out;
  uint64_t out_cap;
  uint32_t* status;
  uint32_t one;                  // always 1 (the MD5 kernels' opaque multiplier)
  unsigned long long* rejected;  // count: djb2 candidates dropped by the byte comparison (or null)
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar,
                                          uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::
          "r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(policy)
      : "memory");
}

// The one-word Bloom filter of a fragment table: a key's word comes from w, its bits from b (both
// 32 bits, see the functions of that name below).
//
// KEYS is the table's class (frag_key_class). A djb2-64 key is represented by g, the low word of h less
// the initial value's share (what the scan rolls), spread by two odd multipliers, in the largest
// tables by both words of it. An MD5 key is represented by its first word, which is final three
// operations before the end of the last block: the filter's bits from the third word, the block from
// the fourth, needed two of these three for every window (1.347 ms for 256 MiB then, 1.336 so). 32
// bits tell keys apart while these are few; 2^26 keys have 2^25 words, 7 bits are left to tell the
// keys of a word apart, and by arithmetic one window in thirty passes instead of one in a hundred
// and fifty. So the largest tables take the bits from the fourth word.
struct FragFilterKey {
  uint32_t w, b;
};

template <int SIG>
__device__ __forceinline__ uint32_t frag_bloom_word(uint32_t w, uint32_t mask) {
  if constexpr (SIG == kSigDjb2) return __umulhi(w, mask + 1u);
  return w & mask;
}

// The key's bits of its word: three bit numbers, for djb2-64 (where the test is off the scan's
// inner loop) five, each taken mod 32: the top bits of b first.
template <int SIG>
constexpr int kFragBloomBits = SIG == kSigDjb2 ? 5 : 3;

__device__ __forceinline__ uint32_t frag_bloom_bit(uint32_t b, int k) { return b >> (27 - 5 * k); }

template <int SIG>
__device__ __forceinline__ bool frag_bloom_hit(uint32_t v, uint32_t b) {
  uint32_t t = 1u;
#pragma unroll
  for (int k = 0; k < kFragBloomBits<SIG>; k++) t &= __funnelshift_r(v, 0u, frag_bloom_bit(b, k));
  return t != 0u;
}

template <int KEYS>
using FragRoll = typename std::conditional<KEYS == kFragMostKeys, uint64_t, uint32_t>::type;

// g: h less the initial value's share, its low word unless KEYS is kFragMostKeys.
template <int KEYS>
__device__ __forceinline__ FragFilterKey frag_djb2_filter_key(FragRoll<KEYS> g) {
  if constexpr (KEYS == kFragMostKeys) {
    const uint32_t lo = (uint32_t)g, hi = (uint32_t)(g >> 32);
    return {(uint32_t)((g * 0x9E3779B97F4A7C15ull) >> 32) + 0x7F4A7C15u, lo * 0x85EBCA77u + hi * 0x9E3779B1u + 0x27D4EB2Fu};
  } else {
    return {g * 0x9E3779B1u + 0x7F4A7C15u, g * 0x85EBCA77u + 0x27D4EB2Fu};  // g = 0: zero windows
  }
}

template <int KEYS>
__device__ __forceinline__ FragFilterKey frag_md5_filter_key(uint32_t d0, uint32_t d3) {
  if constexpr (KEYS == kFragMostKeys) return {d0, d3};
  return {d0, d0 * 0x9E3779B1u};  // the top bits: d0's low ones are the word's number
}

// The shared-memory filter of a djb2 fragment table: bits of the word that the top 15 bits of g
// select, two from the low ten bits of g, or one where there are many keys (at 2^20 keys two bits
// pass 0.75 of the windows, one 0.63). Both bits are set for 0.09 of the windows at 173,751 keys,
// against 0.15 for one bit.
__device__ __forceinline__ uint32_t frag_l1_word(uint32_t g) { return g >> 17; }
template <int KEYS>
__device__ __forceinline__ uint32_t frag_l1_bits(uint32_t g) {
  return (1u << (g & 31)) | (KEYS == kFragFewKeys ? 1u << ((g >> 5) & 31) : 0u);
}
template <int KEYS>
__device__ __forceinline__ uint32_t frag_l1_hit(uint32_t v, uint32_t g) {
  return __funnelshift_r(v, 0u, g) & (KEYS == kFragFewKeys ? __funnelshift_r(v, 0u, g >> 5) : 1u) & 1u;
}

// djb2-64 of consecutive windows w0, w0 + 1, ... (ws: 32-bit words in shared memory), rolled:
// first() computes window w0 from its 16 words, then next(x, i) moves to window w0 + i (called for
// i = 1, 2, ... in order) with one new word. P holds the Horner values of the current window's
// words, g = h - 5381 * 33^64. U: uint64_t, or uint32_t for the low word of g alone.
template <class U>
struct Djb2Roll {
  uint32_t P[16];
  U g;
  __device__ __forceinline__ void first(const uint32_t* ws, uint32_t w0) {
    g = 0;
#pragma unroll
    for (int q = 0; q < 16; q++) {
      P[q] = horner33(ws[w0 + q]);
      g = g * (U)kD33x4 + P[q];
    }
  }
  // x: the new window's last word (ws[w0 + i + 15])
  __device__ __forceinline__ void next(uint32_t x, int i) {
    const uint32_t pin = horner33(x);
    g = g * (U)kD33x4 + (P[(i - 1) & 15] * (U)(0 - kD33x64) + pin);
    P[(i - 1) & 15] = pin;
  }
};

// Key words of the window whose 16 words start at x, computed directly.
template <int SIG>
__device__ __forceinline__ void frag_key(const uint32_t* x, uint32_t (&d)[4], uint32_t one) {
  uint32_t X[16];
#pragma unroll
  for (int q = 0; q < 16; q++) X[q] = x[q];
  if constexpr (SIG == kSigDjb2) {
    frag64_words(djb2_block(5381ull, X), d);
  } else {
    md5_init(d);
    md5_compress<0>(d, X, one);
    if constexpr (SIG == kSigMd5) md5_compress_block_padding(d, one);
  }
}

// The 64 bytes at x (4-byte aligned) against a master fragment (16-byte aligned).
__device__ __forceinline__ bool frag_equal(const uint32_t* x, const uint8_t* m) {
  const uint4* y = reinterpret_cast<const uint4*>(m);
  uint32_t diff = 0;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const uint4 v = __ldg(y + q);
    diff |= (x[4 * q] ^ v.x) | (x[4 * q + 1] ^ v.y) | (x[4 * q + 2] ^ v.z) | (x[4 * q + 3] ^ v.w);
  }
  return diff == 0;
}

// Candidate windows of this thread (bit i: window w0 + i passed the filters that the table has). n_valid: the thread's windows inside the
// image. l1: the first filter (rolled kernels only). ws is the warp's tile; the waiting windows of the
// rolled kernel for few keys overwrite parts of it (FragGeom::kQueue).
//
// Not rolled (MD5): the hash is all of the cost (126 or 61 operations a window), so a window that equals
// the one before it (fills; patterns of four bytes) is not hashed again. The lanes mark these (17
// equal words), the others are listed and dealt out evenly over the warp, a candidate sets its bit in
// its lane's mask, and the windows after it that equal it are candidates too. Where no two words at
// the multiples of 16 and after are equal there is no such run, and the lanes hash their own windows.
// 256 MiB of which 15% of the sectors are zeros 1,336 to 1,227 us, half of it zeros 1,312 to 728; random
// bytes 1,342 to 1,347 (without the padding block 790 to 804).
//
// Rolled: the cost is instructions, not memory. A window takes one shared-memory word, two dp2a,
// two multiply-adds and the filter (word address, load, two shifts by the low bits of g, which wrap
// by themselves); its random load, 3.6 shared-memory cycles on average, sets the pace. The windows
// that pass (one in twelve at 173,751 keys) only store their g; their Bloom words are requested
// afterwards. 1 GiB image, count kernel: the loop alone takes 225 us (shared memory 85% busy), the
// Bloom words 105 more, the lookups 55: 388 us, against 800 with 64-bit h, one filter bit and the
// Bloom test inside the loop, where its dozen instructions are executed for every window because
// some lane nearly always has one to test. Dealing the waiting windows out evenly over the warp
// (a scan and searches by shuffles) took 392 us: shuffles use the same pipe.
// A window with the g of the window before it (fills, patterns of four bytes) shares that one's
// entry, so such runs need one place; a lane with more passing windows than places sends the rest
// on unfiltered. The stores are predicated by hand (a branch per window cost more than they do),
// and each word is read a window ahead because no load may move past them.
//
// That holds while few windows pass the first filter. It has 2^20 bits whatever the table's size: at
// 500,000 keys 0.38 of the windows pass and at 2^20 three of four, most lanes then have more than eight
// of them, and each one sent on costs 16 words, the whole hash and a slot (1,564 and 6,350 us). With
// many keys every window that passes asks for its Bloom word in the loop, six ahead of their tests,
// and the tile stays as it is: 692 and 1,165 us. The most keys: nearly every window passes, so
// the first filter is not looked at, and the Bloom words, from L2 and DRAM, are all of the cost. What
// matters then is an even stream of requests: words asked for in rounds of 4, 8 and 23 took 3,780,
// 3,835 and 4,370 us at 2^25 keys, four or six ahead 3,522 and 3,529, twelve ahead 3,772.
template <int SIG, int KEYS>
__device__ __forceinline__ uint32_t frag_candidates(const FragParams& p, uint32_t* ws, uint32_t w0, uint32_t n_valid,
                                                    const uint32_t* l1, uint16_t* list, uint32_t* masks) {
  using G = FragGeom<SIG>;
  if constexpr (G::kRolled && KEYS != kFragFewKeys) {
    const uint32_t* const bloom = reinterpret_cast<const uint32_t*>(p.tab.bloom);
    Djb2Roll<FragRoll<KEYS>> roll;
    uint32_t cand = 0;
    constexpr int kAhead = 6;
    uint32_t v[kAhead], bits[kAhead];
#pragma unroll
    for (int i = 0; i < G::kWPT + kAhead; i++) {
      if (i >= kAhead) {  // before window i takes its place
        const int q = i - kAhead;
        if (frag_bloom_hit<SIG>(v[q % kAhead], bits[q % kAhead])) cand |= 1u << q;
      }
      if (i < G::kWPT) {
        if (i == 0) roll.first(ws, w0);
        else roll.next(ws[w0 + i + 15], i);
        const FragFilterKey key = frag_djb2_filter_key<KEYS>(roll.g);
        bool pass = true;
        if constexpr (KEYS != kFragMostKeys) pass = frag_l1_hit<KEYS>(l1[frag_l1_word(roll.g)], roll.g);
        bits[i % kAhead] = key.b;
        v[i % kAhead] = 0u;
        if (pass) v[i % kAhead] = p.tab.use_bloom ? __ldg(bloom + frag_bloom_word<SIG>(key.w, p.tab.bloom_mask)) : ~0u;
      }
    }
    // windows past the image's end come last
    return n_valid < (uint32_t)G::kWPT ? cand & ((1u << n_valid) - 1u) : cand;
  } else if constexpr (G::kRolled) {
    const uint32_t queue = smem_addr(ws + w0 + 15), queue_end = queue + 4u * G::kQueue;
    Djb2Roll<uint32_t> roll;
    uint32_t pass = 0, fresh = 0, at = queue, x = 0, before = 0;
#pragma unroll
    for (int i = 0; i < G::kWPT; i++) {
      if (i == 0) {
        roll.first(ws, w0);
        before = ~roll.g;
      } else {
        before = roll.g;
        roll.next(x, i);
      }
      if (i + 1 < G::kWPT) x = ws[w0 + i + 16];
      asm volatile(
          "{\n\t.reg .pred hit, first, room;\n\t"
          "setp.ne.u32 hit, %3, 0;\n\t"
          "setp.ne.and.u32 first, %4, %5, hit;\n\t"
          "setp.lt.and.u32 room, %0, %6, first;\n\t"
          "@room st.shared.u32 [%0], %4;\n\t"
          "@first add.u32 %0, %0, 4;\n\t"
          "@first or.b32 %1, %1, %7;\n\t"
          "@hit or.b32 %2, %2, %7;\n\t}"
          : "+r"(at), "+r"(fresh), "+r"(pass)
          : "r"(frag_l1_hit<KEYS>(l1[frag_l1_word(roll.g)], roll.g)), "r"(roll.g), "r"(before), "r"(queue_end), "r"(1u << i)
          : "memory");
    }
    // windows past the image's end come last
    if (n_valid < (uint32_t)G::kWPT) {
      pass &= (1u << n_valid) - 1u;
      fresh &= (1u << n_valid) - 1u;
    }
    if (!p.tab.use_bloom) return pass;
    const uint32_t* bloom = reinterpret_cast<const uint32_t*>(p.tab.bloom);
    const uint32_t* const waiting = ws + w0 + 15;
    const uint32_t same = pass ^ fresh, n = min((uint32_t)__popc(fresh), (uint32_t)G::kQueue);
    uint32_t cand = 0;
    for (uint32_t k = 0; k < n; k += 2) {  // two requests at a time
      const bool two = k + 1 < n;
      const FragFilterKey k0 = frag_djb2_filter_key<KEYS>(waiting[k]);
      const FragFilterKey k1 = frag_djb2_filter_key<KEYS>(two ? waiting[k + 1] : 0u);
      const uint32_t v0 = __ldg(bloom + frag_bloom_word<SIG>(k0.w, p.tab.bloom_mask));
      const uint32_t v1 = two ? __ldg(bloom + frag_bloom_word<SIG>(k1.w, p.tab.bloom_mask)) : 0u;
      const uint32_t b0 = fresh & (0u - fresh);
      fresh ^= b0;
      if (frag_bloom_hit<SIG>(v0, k0.b)) cand |= b0;
      if (two) {
        const uint32_t b1 = fresh & (0u - fresh);
        fresh ^= b1;
        if (frag_bloom_hit<SIG>(v1, k1.b)) cand |= b1;
      }
    }
    cand |= fresh;
    // the windows after a candidate that share its entry: a carry through each run of them
    return cand | (((same + (same & (cand << 1))) ^ same) & same);
  } else {
    constexpr uint32_t kFull = 0xFFFFFFFFu;
    constexpr uint32_t kWords = G::kWPT + 15;  // of this lane's windows
    const uint32_t lane = w0 / G::kWPT;
    uint32_t same = 0;  // bit i: window w0 + i equals the one before it
    // 17 equal words have one among them whose number is a multiple of 16, and the one after it
    bool some = false;
    for (uint32_t k = (w0 + 15u) & ~15u; k + 1 < w0 + kWords; k += 16) some |= ws[k] == ws[k + 1];
    uint32_t rounds = n_valid, total = 0;
    bool listed = false;
    if (__any_sync(kFull, some)) {
      // equal: bit k, word k + 1 is word k; window i is the one before it if bits i - 1 .. i + 14 are set
      uint32_t lo = 0, hi = 0, before = ws[w0];
#pragma unroll
      for (uint32_t k = 0; k + 1 < kWords; k++) {
        const uint32_t x = ws[w0 + k + 1];
        if (x == before) {
          if (k < 32) lo |= 1u << (k & 31);
          else hi |= 1u << (k & 31);
        }
        before = x;
      }
      uint64_t equal = (uint64_t)hi << 32 | lo;
#pragma unroll
      for (int d = 1; d < 16; d <<= 1) equal &= equal >> d;
      const uint32_t valid = (uint32_t)((1ull << n_valid) - 1u);
      same = (uint32_t)equal << 1 & valid;
      const uint32_t need = valid ^ same;
      uint32_t at = __popc(need);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, at, d);
        if (lane >= (uint32_t)d) at += v;
      }
      total = __shfl_sync(kFull, at, 31);
      at -= __popc(need);
      listed = (total + 31) / 32 < __reduce_max_sync(kFull, n_valid);
      if (listed) {
        rounds = (total + 31 - lane) / 32;
        masks[lane] = 0;
#pragma unroll
        for (uint32_t i = 0; i < (uint32_t)G::kWPT; i++)
          if (need >> i & 1u) list[at++] = (uint16_t)(w0 + i);
        __syncwarp();
      }
    }
    uint32_t cand = 0;
#pragma unroll 1
    for (uint32_t r = 0; r < rounds; r++) {
      const uint32_t w = listed ? list[32 * r + lane] : w0 + r;
      uint32_t d[4];
      frag_key<SIG>(ws + w, d, p.one);
      const FragFilterKey key = frag_md5_filter_key<KEYS>(d[0], d[3]);
      if (!p.tab.use_bloom || frag_bloom_hit<SIG>(__ldg(reinterpret_cast<const uint32_t*>(p.tab.bloom) +
                                                        frag_bloom_word<SIG>(key.w, p.tab.bloom_mask)),
                                                  key.b)) {
        if (listed) atomicOr(masks + w / G::kWPT, 1u << (w % G::kWPT));
        else cand |= 1u << r;
      }
    }
    if (!listed) return cand;
    __syncwarp();
    cand = masks[lane];
    return cand | (((same + (same & (cand << 1))) ^ same) & same);
  }
}

// The image of a tile.
template <bool MULTI>
__device__ __forceinline__ const FragImage& frag_image(const FragParams& p, uint64_t tile) {
  if constexpr (!MULTI) return p.images.in[0];
  const FragImage* const im = p.images.get();
  uint32_t lo = 0, hi = p.images.n;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) >> 1;
    if (im[mid].tile_base <= tile) lo = mid; else hi = mid;
  }
  return im[lo];
}

// The 16 words of this thread's window w0 + i of the image's tile: in the staged tile, or, where that may
// be overwritten, in the image.
template <int SIG, int KEYS>
__device__ __forceinline__ const uint32_t* frag_words(const FragImage& im, uint64_t tile, const uint32_t* ws,
                                                      uint32_t w) {
  if constexpr (FragGeom<SIG>::kRolled && KEYS == kFragFewKeys)
    return reinterpret_cast<const uint32_t*>(im.data) + (tile * FragGeom<SIG>::kTileWin + w);
  return ws + w;
}

// One candidate window per lane (has; x: its words) looked up; returns the triples it yields
// (postings, confirmed byte for byte for djb2) and its posting range. The lanes of the warp
// compare the postings of a window that has several together: a header that hundreds of files
// share has hundreds. Every lane of the warp calls it.
template <int SIG, int LAYOUT>
__device__ __forceinline__ uint32_t frag_resolve(const FragParams& p, const uint32_t* x, bool has, uint32_t& post_off,
                                                 uint32_t& post_cnt) {
  post_off = 0;
  post_cnt = 0;
  if (has) {
    uint32_t d[4];
    frag_key<SIG>(x, d, p.one);
    post_cnt = LAYOUT == kLayoutSorted ? sorted_probe(p.tab, d[0], d[1], d[2], d[3], 0u, post_off)
                                       : table_probe(p.tab, d[0], d[1], d[2], d[3], 0u, post_off);
  }
  if constexpr (!sig_is_weak(SIG)) return post_cnt;
  uint32_t n = 0;
  if (post_cnt == 1u) n = frag_equal(x, p.tab.confirm + (uint64_t)post_off * 64) ? 1u : 0u;
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t several = __ballot_sync(0xFFFFFFFFu, post_cnt > 1u); several; several &= several - 1) {
    const int src = __ffs(several) - 1;
    const uint32_t* xs = reinterpret_cast<const uint32_t*>(
        __shfl_sync(0xFFFFFFFFu, reinterpret_cast<uintptr_t>(x), src));
    const uint32_t off = __shfl_sync(0xFFFFFFFFu, post_off, src), cnt = __shfl_sync(0xFFFFFFFFu, post_cnt, src);
    uint32_t k = 0;
    for (uint32_t q = lane; q < cnt; q += 32) k += frag_equal(xs, p.tab.confirm + (uint64_t)(off + q) * 64) ? 1u : 0u;
    k = __reduce_add_sync(0xFFFFFFFFu, k);
    if ((int)lane == src) n = k;
  }
  return n;
}

// Triples of this thread's candidate windows; hits: the windows with any; *rejected adds the
// candidates that the byte comparison dropped. Every lane of the warp calls it.
template <int SIG, int LAYOUT, int KEYS>
__device__ __forceinline__ uint64_t frag_thread_count(const FragParams& p, const FragImage& im, uint64_t tile,
                                                      const uint32_t* ws, uint32_t w0, uint32_t cand, uint32_t& hits, uint32_t* rejected) {
  uint64_t n = 0;
  hits = 0;
  while (__any_sync(0xFFFFFFFFu, cand != 0)) {
    const bool has = cand != 0;
    const uint32_t i = has ? (uint32_t)__ffs(cand) - 1u : 0u;
    cand &= cand - 1;
    uint32_t off, cnt;
    const uint32_t k = frag_resolve<SIG, LAYOUT>(p, frag_words<SIG, KEYS>(im, tile, ws, w0 + i), has, off, cnt);
    n += k;
    if (k) hits |= 1u << i;
    *rejected += cnt - k;
  }
  return n;
}

__device__ __forceinline__ uint64_t shfl_up_u64(uint64_t v, int d) {
  const uint32_t lo = __shfl_up_sync(0xFFFFFFFFu, (uint32_t)v, d);
  const uint32_t hi = __shfl_up_sync(0xFFFFFFFFu, (uint32_t)(v >> 32), d);
  return ((uint64_t)hi << 32) | lo;
}

// Warp-wide exclusive scan of one u64 per lane; *total receives the sum (every lane).
__device__ __forceinline__ uint64_t warp_exclusive_u64(uint64_t v, uint64_t* total) {
  const int lane = threadIdx.x & 31;
  uint64_t incl = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t x = shfl_up_u64(incl, d);
    if (lane >= d) incl += x;
  }
  const uint32_t lo = __shfl_sync(0xFFFFFFFFu, (uint32_t)incl, 31);
  const uint32_t hi = __shfl_sync(0xFFFFFFFFu, (uint32_t)(incl >> 32), 31);
  *total = ((uint64_t)hi << 32) | lo;
  return incl - v;
}

// Lane 0: issue the image's tile `tile` into the buffer at smem address dst (completion on bar).
template <int SIG>
__device__ __forceinline__ void frag_issue(const FragImage& im, uint64_t tile, uint32_t dst, uint32_t bar,
                                           uint64_t policy) {
  using G = FragGeom<SIG>;
  const uint64_t start = tile * G::kTileStep;
  const uint64_t left = im.n_bytes - start;
  const uint32_t avail = left < G::kTileBytes ? (uint32_t)left : G::kTileBytes;
  const uint32_t bulk = avail & ~15u;
  mbar_arrive_expect_tx(bar, bulk);
  if (bulk) bulk_load(dst, im.data + start, bulk, bar, policy);
}

// The bytes of the tile past its last whole 16-byte chunk (the bulk copy moves whole chunks
// only), with plain loads by the warp's lanes; only the image's last tile has any. Ends with a
// warp barrier.
template <int SIG>
__device__ __forceinline__ void frag_tail(const FragImage& im, uint64_t tile, uint8_t* buf) {
  using G = FragGeom<SIG>;
  const uint64_t start = tile * G::kTileStep;
  const uint64_t left = im.n_bytes - start;
  const uint32_t avail = left < G::kTileBytes ? (uint32_t)left : G::kTileBytes;
  const uint32_t b = (avail & ~15u) + (threadIdx.x & 31);
  if (b < avail) buf[b] = im.data[start + b];
  __syncwarp();
}

template <int SIG>
__device__ __forceinline__ uint32_t frag_valid(const FragImage& im, uint64_t tile, uint32_t w0) {
  using G = FragGeom<SIG>;
  const uint64_t k0 = tile * G::kTileWin + w0;
  if (k0 >= im.n_windows) return 0u;
  const uint64_t left = im.n_windows - k0;
  return left < (uint64_t)G::kWPT ? (uint32_t)left : (uint32_t)G::kWPT;
}

// MULTI: several images, one after another in tile numbers; a tile's image is found by search. (With a
// launch per image, small ones ran one after another, each on a few SMs, and as many emit launches behind
// them: 200 images of 64 KiB without a match took 2,460 us, MD5 10,470; in one go 256 and 341.) For one
// image its parameters are constants of the launch, which the kernels' registers are laid out for.
template <int SIG, int LAYOUT, int KEYS, bool MULTI>
__global__ void __launch_bounds__(FragGeom<SIG>::kThreads, FragGeom<SIG>::kMinBlocks)
    frag_count_kernel(const __grid_constant__ FragParams p) {
  using G = FragGeom<SIG>;
  extern __shared__ __align__(128) uint8_t fsm[];
  __shared__ __align__(8) uint64_t bars[G::kWarps + 1];  // one per warp, the shared-memory filter
  __shared__ uint32_t abort_flag[G::kWarps + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t* l1 = G::kL1 ? reinterpret_cast<const uint32_t*>(fsm + G::kL1Off) : nullptr;
  uint8_t* buf = fsm + warp * G::kTileBytes;
  uint32_t* const masks = G::kRolled ? nullptr : reinterpret_cast<uint32_t*>(fsm + G::kL1Off + warp * G::kListBytes);
  uint16_t* const list = G::kRolled ? nullptr : reinterpret_cast<uint16_t*>(masks + 32);
  const uint32_t bar = smem_addr(&bars[warp]);
  const uint32_t bar_l1 = smem_addr(&bars[G::kWarps]);
  if (tid == 0) {
    for (int b = 0; b < G::kWarps + 1; b++) mbar_init(smem_addr(&bars[b]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid <= G::kWarps) abort_flag[tid] = 0;
  __syncthreads();
  const uint64_t policy = l2_evict_first_policy();
  const uint64_t n_warps = (uint64_t)gridDim.x * G::kWarps;
  const uint64_t first = (uint64_t)blockIdx.x * G::kWarps + warp;
  // The warp's i-th tile completes phase i of its buffer's barrier; lane 0 issues the next tile when
  // every lane is done with the buffer (the other warps of the SM cover the copy).
  if (tid == 0 && G::kL1) {
    mbar_arrive_expect_tx(bar_l1, kFragL1Bytes);
    bulk_load(smem_addr(fsm + G::kL1Off), p.tab.frag_l1, kFragL1Bytes, bar_l1, policy);
  }
  const auto issue = [&](uint64_t tile) {
    const FragImage& im = frag_image<MULTI>(p, tile);
    frag_issue<SIG>(im, tile - (MULTI ? im.tile_base : 0ull), smem_addr(buf), bar, policy);
  };
  if (lane == 0 && first < p.n_tiles) issue(first);
  bool ok = true;
  if constexpr (G::kL1) ok = mbar_wait(bar_l1, 0u, &abort_flag[G::kWarps], p.status);
  bool aborted = !__syncthreads_and(ok);  // the only block-wide barrier: the filter is in place
  uint64_t i = 0;
  for (; !aborted; i++) {
    const uint64_t tile = first + i * n_warps;
    if (tile >= p.n_tiles) break;
    ok = mbar_wait(bar, (uint32_t)i & 1u, &abort_flag[warp], p.status);
    if (!__all_sync(0xFFFFFFFFu, ok)) {
      aborted = true;
      break;
    }
    const FragImage& im = frag_image<MULTI>(p, tile);
    const uint64_t local = tile - (MULTI ? im.tile_base : 0ull);
    if ((local + 1) * G::kTileStep + 64 > im.n_bytes) frag_tail<SIG>(im, local, buf);  // warp-uniform
    uint32_t* ws = reinterpret_cast<uint32_t*>(buf);
    const uint32_t w0 = (uint32_t)lane * G::kWPT;
    const uint32_t cand = frag_candidates<SIG, KEYS>(p, ws, w0, frag_valid<SIG>(im, local, w0), l1, list, masks);
    uint32_t rej = 0;
    uint32_t hits;
    uint64_t n = frag_thread_count<SIG, LAYOUT, KEYS>(p, im, local, ws, w0, cand, hits, &rej);
    if (sig_is_weak(SIG) && rej && p.rejected) atomicAdd(p.rejected, (unsigned long long)rej);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) n += __shfl_xor_sync(0xFFFFFFFFu, n, d);
    if (n) {  // the sum over the warp
      uint32_t q = 0;
      if (lane == 0) q = atomicAdd(p.n_hit_tiles, 1u);
      q = __shfl_sync(0xFFFFFFFFu, q, 0);
      if (lane == 0) p.hit_tiles[q] = (uint32_t)tile;
      if (q < p.mask_cap) p.hit_masks[32ull * q + lane] = hits;
    }
    __syncwarp();  // every lane is done with the buffer
    if (lane == 0) {
      p.tile_ntrip[tile] = n;
      const uint64_t next = tile + n_warps;
      if (next < p.n_tiles) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        issue(next);
      }
    }
    __syncwarp();
  }
  if (aborted && lane == 0) {
    // The filter (lane 0 of warp 0) and this warp's tile may have copies issued and not waited for:
    // let them land, each wait bounded, before shared memory goes away.
    volatile uint32_t never = 0;
    if (G::kL1 && tid == 0) mbar_wait(bar_l1, 0u, &never, p.status);
    if (first + i * n_warps < p.n_tiles) mbar_wait(bar, (uint32_t)i & 1u, &never, p.status);
  }
}

// Triple `pos` of the output: window k and posting `post`.
__device__ __forceinline__ void frag_put(const FragParams& p, uint64_t pos, uint64_t k, uint32_t post) {
  if (pos < p.out_cap) {
    const uint2 e = __ldg(p.tab.postings + post);
    p.out[pos] = MatchOut{k, e.x, e.y};
  } else {
    atomicOr(p.status, kStOverflow);
  }
}

// A warp per listed tile: its windows with triples are numbered in window order (a lane's windows
// follow one another) and taken 32 at a time, one per lane, so that the dependent loads of 32 of
// them (words, slot, confirmation, posting) are in flight together. Bound by that latency. Without room
// for the triples of all images nothing is looked up and the overflow is flagged once.
constexpr int kEmitThreads = 256;

template <int SIG, int LAYOUT>
__global__ void __launch_bounds__(kEmitThreads) frag_emit_kernel(const __grid_constant__ FragParams p) {
  using G = FragGeom<SIG>;
  if (*(volatile const uint32_t*)p.status & (kStTimeout | kStProbeBound | kStBadTable)) return;
  if (*p.total > p.out_cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(p.status, kStOverflow);
    return;
  }
  constexpr uint32_t kFull = 0xFFFFFFFFu;
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t n_list = *(volatile const uint32_t*)p.n_hit_tiles;
  const uint32_t n_warps = gridDim.x * (kEmitThreads / 32);
  for (uint32_t j = blockIdx.x * (kEmitThreads / 32) + (threadIdx.x >> 5); j < n_list; j += n_warps) {
    const uint64_t numbered = p.hit_tiles[j];
    const FragImage& im = frag_image<true>(p, numbered);
    const uint64_t tile = numbered - im.tile_base;
    // beyond the masks' room every window is looked up
    const uint32_t valid = frag_valid<SIG>(im, tile, lane * G::kWPT);
    const uint32_t mask = j < p.mask_cap ? p.hit_masks[32ull * j + lane] : (uint32_t)((1ull << valid) - 1u);
    uint64_t at = p.tile_off[numbered];
    const uint32_t n = (uint32_t)__popc(mask);
    uint32_t first = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(kFull, first, d);
      if (lane >= (uint32_t)d) first += v;
    }
    const uint32_t total = __shfl_sync(kFull, first, 31);
    first -= n;
    for (uint32_t e0 = 0; e0 < total; e0 += 32) {
      // window number e: the k-th window of the last lane whose first number is at or before e
      const uint32_t e = e0 + lane;
      uint32_t src = 0;
#pragma unroll
      for (uint32_t step = 16; step > 0; step >>= 1)
        if (__shfl_sync(kFull, first, src + step) <= e) src += step;
      const bool has = e < total;
      uint32_t k = e - __shfl_sync(kFull, first, src);
      uint32_t m = __shfl_sync(kFull, mask, src);
      if (!has) k = 0;
      for (; k > 0; k--) m &= m - 1;
      const uint64_t w = tile * G::kTileWin + src * G::kWPT + (has ? (uint32_t)__ffs(m) - 1u : 0u);
      const uint32_t* x = reinterpret_cast<const uint32_t*>(im.data) + w;
      uint32_t off, cnt;
      const uint32_t put = frag_resolve<SIG, LAYOUT>(p, x, has, off, cnt);
      uint64_t sum;
      const uint64_t pos = at + warp_exclusive_u64(put, &sum);
      at += sum;
      if (cnt == 1u && put == 1u) frag_put(p, pos, w, off);
      // the postings of a window with several, 32 at a time
      for (uint32_t several = __ballot_sync(kFull, cnt > 1u); several; several &= several - 1) {
        const int from = __ffs(several) - 1;
        const uint32_t* xs = reinterpret_cast<const uint32_t*>(__shfl_sync(kFull, reinterpret_cast<uintptr_t>(x), from));
        const uint32_t o = __shfl_sync(kFull, off, from), c = __shfl_sync(kFull, cnt, from);
        const uint64_t ww = __shfl_sync(kFull, (unsigned long long)w, from);
        uint64_t to = __shfl_sync(kFull, (unsigned long long)pos, from);
        for (uint32_t q0 = 0; q0 < c; q0 += 32) {
          const uint32_t q = q0 + lane;
          const bool equal = q < c && (!sig_is_weak(SIG) || frag_equal(xs, p.tab.confirm + (uint64_t)(o + q) * 64));
          const uint32_t who = __ballot_sync(kFull, equal);
          if (equal) frag_put(p, to + __popc(who & ((1u << lane) - 1u)), ww, o + q);
          to += __popc(who);
        }
      }
    }
  }
}

// The signature of every window of an image, 16 bytes per window, through the count kernel's
// own arithmetic: the rolled djb2 of Djb2Roll (each lane's first window computed directly and the
// others rolled), or frag_key for MD5. For djb2 the 16 bytes are the
// table key words (h, then the mixing word of frag64_words). One warp per tile, staged with
// plain loads; a test and diagnostic path, not the scan. Its tiles are its own: bound by the 16 bytes
// written per window, a warp's stores a tile's lane apart, it takes 17 djb2 windows a lane better than the
// count kernel's 23 (64 KiB 8.5 against 10.6 us, 64 MiB 120 against 134, 256 MiB 439 against 465).
template <int SIG>
struct FragSigTile {
  static constexpr int kWPT = SIG == kSigDjb2 ? 17 : FragGeom<SIG>::kWPT;  // windows per lane (odd)
  static constexpr uint32_t kWin = 32 * kWPT;
  static constexpr uint32_t kStep = kWin * kFragStride;
  static constexpr uint32_t kBytes = kStep + 64;
};

template <int SIG>
__global__ void __launch_bounds__(256) frag_window_sig_kernel(const uint8_t* image, uint64_t n_bytes,
                                                              uint64_t n_windows, uint64_t n_tiles, uint4* out,
                                                              uint32_t one) {
  using G = FragSigTile<SIG>;
  extern __shared__ __align__(128) uint8_t fsm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* ws = reinterpret_cast<uint32_t*>(fsm + warp * G::kBytes);
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  for (uint64_t tile = (uint64_t)blockIdx.x * (blockDim.x >> 5) + warp; tile < n_tiles; tile += warps) {
    const uint64_t start = tile * G::kStep;
    for (uint32_t j = lane; j < G::kBytes / 4; j += 32) {
      const uint64_t b = start + 4ull * j;
      uint32_t v = 0;
      if (b + 4 <= n_bytes) {
        v = *reinterpret_cast<const uint32_t*>(image + b);
      } else {
        for (uint32_t q = 0; q < 4; q++)
          if (b + q < n_bytes) v |= (uint32_t)image[b + q] << (8 * q);
      }
      ws[j] = v;
    }
    __syncwarp();
    const uint32_t w0 = (uint32_t)lane * G::kWPT;
    const uint64_t k0 = tile * G::kWin + w0;
    if constexpr (SIG == kSigDjb2) {
      Djb2Roll<uint64_t> roll;
#pragma unroll
      for (int i = 0; i < G::kWPT; i++) {
        if (i == 0) roll.first(ws, w0);
        else roll.next(ws[w0 + i + 15], i);
        uint32_t d[4];
        frag64_words(roll.g + kDjbInit, d);
        if (k0 + i < n_windows) out[k0 + i] = make_uint4(d[0], d[1], d[2], d[3]);
      }
    } else {
      for (int i = 0; i < G::kWPT; i++) {
        if (k0 + i >= n_windows) break;
        uint32_t d[4];
        frag_key<SIG>(ws + w0 + i, d, one);
        out[k0 + i] = make_uint4(d[0], d[1], d[2], d[3]);
      }
    }
    __syncwarp();
  }
}

// ------------------------------------------------------------------------ master side
// Key words of every master fragment (64 bytes each, 16-byte aligned) and its exclusion flag
// (all 64 bytes equal).
template <int SIG>
__global__ void frag_digest_kernel(const uint8_t* arena, uint64_t n, uint4* dig, uint8_t* trivial, uint32_t one) {
  for (uint64_t m = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (uint64_t)gridDim.x * blockDim.x) {
    const uint4* src = reinterpret_cast<const uint4*>(arena + m * 64);
    uint32_t X[16];
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint4 v = src[q];
      X[4 * q] = v.x;
      X[4 * q + 1] = v.y;
      X[4 * q + 2] = v.z;
      X[4 * q + 3] = v.w;
    }
    const uint32_t rep = (X[0] & 0xFFu) * 0x01010101u;
    uint32_t diff = 0;
#pragma unroll
    for (int q = 0; q < 16; q++) diff |= X[q] ^ rep;
    uint32_t d[4];
    if constexpr (SIG == kSigDjb2) {
      frag64_words(djb2_block(5381ull, X), d);
    } else {
      md5_init(d);
      md5_compress<3>(d, X, one);
      if constexpr (SIG == kSigMd5) md5_compress_block_padding(d, one);
    }
    dig[m] = make_uint4(d[0], d[1], d[2], d[3]);
    trivial[m] = diff == 0u ? 1 : 0;
  }
}

// The filters of a fragment table from its occupied slots: the one-word Bloom filter (none when
// words is null) and the shared-memory filter.
template <int SIG, int KEYS>
__global__ void frag_bloom_kernel(const uint4* slots, uint32_t n_slots, uint32_t* words, uint32_t mask,
                                  uint32_t* l1) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_slots; i += gridDim.x * blockDim.x) {
    if (slots[2ull * i + 1].y == 0u) continue;
    const uint4 d = slots[2ull * i];
    const uint64_t g = ((uint64_t)d.y << 32 | d.x) - kDjbInit;  // djb2
    if (words) {
      FragFilterKey key;
      if constexpr (SIG == kSigDjb2) key = frag_djb2_filter_key<KEYS>((FragRoll<KEYS>)g);
      else key = frag_md5_filter_key<KEYS>(d.x, d.w);
      uint32_t bits = 0;
      for (int k = 0; k < kFragBloomBits<SIG>; k++) bits |= 1u << (frag_bloom_bit(key.b, k) & 31);
      atomicOr(words + frag_bloom_word<SIG>(key.w, mask), bits);
    }
    if (SIG == kSigDjb2) atomicOr(l1 + frag_l1_word((uint32_t)g), frag_l1_bits<KEYS>((uint32_t)g));
  }
}

// ------------------------------------------------------------------------------ host
namespace {

using KernelFn = const void*;

struct Geom {
  KernelFn count, emit;
  int threads;
  uint32_t tile_win, smem_count;
};

template <int SIG, int LAYOUT, bool MULTI>
KernelFn count_fn(int keys) {
  if (keys == kFragMostKeys) return (KernelFn)frag_count_kernel<SIG, LAYOUT, kFragMostKeys, MULTI>;
  if constexpr (FragGeom<SIG>::kRolled)
    if (keys == kFragManyKeys) return (KernelFn)frag_count_kernel<SIG, LAYOUT, kFragManyKeys, MULTI>;
  return (KernelFn)frag_count_kernel<SIG, LAYOUT, kFragFewKeys, MULTI>;
}

template <int SIG>
Geom geom_t(uint32_t layout, int keys, bool multi) {
  using G = FragGeom<SIG>;
  const bool s = layout == kLayoutSorted;
  const KernelFn count = multi ? s ? count_fn<SIG, kLayoutSorted, true>(keys) : count_fn<SIG, kLayoutHash, true>(keys)
                         : s   ? count_fn<SIG, kLayoutSorted, false>(keys)
                               : count_fn<SIG, kLayoutHash, false>(keys);
  return Geom{count,
              s ? (KernelFn)frag_emit_kernel<SIG, kLayoutSorted> : (KernelFn)frag_emit_kernel<SIG, kLayoutHash>,
              G::kThreads, G::kTileWin, G::kSmemCount};
}

bool geom(int sig, uint32_t layout, int keys, bool multi, Geom* g) {
  switch (sig) {
    case kSigMd5: *g = geom_t<kSigMd5>(layout, keys, multi); return true;
    case kSigMd5NoPad: *g = geom_t<kSigMd5NoPad>(layout, keys, multi); return true;
    case kSigDjb2: *g = geom_t<kSigDjb2>(layout, keys, multi); return true;
    default: return false;
  }
}

struct FragDev {
  bool ready = false;
  int count_blocks[3][2][kFragKeyClasses][2] = {};
};
std::mutex g_frag_mu;
FragDev g_frag_dev[64];

// Shared-memory attributes and resident blocks per SM of every fragment kernel, once per device.
int frag_device(FragDev** out) {
  int dev;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  if (dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_frag_mu);
  FragDev& d = g_frag_dev[dev];
  if (!d.ready) {
    for (int sig = 0; sig < 3; sig++)
      for (int q = 0; q < 4 * kFragKeyClasses; q++) {
        const int l = q & 1, multi = q >> 1 & 1, keys = q >> 2;
        Geom g;
        geom(sig, (uint32_t)l, keys, multi != 0, &g);
        if ((e = cudaFuncSetAttribute(g.count, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)g.smem_count)) !=
            cudaSuccess)
          return (int)e;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&d.count_blocks[sig][l][keys][multi], g.count, g.threads,
                                                               g.smem_count)) != cudaSuccess)
          return (int)e;
        if (d.count_blocks[sig][l][keys][multi] < 1) return (int)cudaErrorInvalidConfiguration;
      }
    d.ready = true;
  }
  *out = &d;
  return 0;
}

FragParams make_params(const TableView& tab, const FragImages& images, uint64_t n_tiles, const FragHits& hits,
                       uint32_t* status) {
  FragParams p;
  memset(&p, 0, sizeof p);
  p.tab = tab;
  p.images = images;
  p.n_tiles = n_tiles;
  p.hit_tiles = hits.tiles;
  p.hit_masks = hits.masks;
  p.mask_cap = (uint32_t)hits.mask_tiles;
  p.n_hit_tiles = hits.count;
  p.status = status;
  p.one = 1u;
  return p;
}

}  // namespace

int frag_key_class(int sig, uint64_t n_keys) {
  // Where the count kernels measured equal on random images, us per scan:
  //   djb2-64, 1 GiB       few     many    most
  //     173,751 keys       368     446
  //     250,000            466     485
  //     300,000            519     472
  //     500,000            1,564   692     1,872
  //     4,194,304          12,607  1,911   1,932
  //     16,777,216                 2,016   1,933
  //     67,108,864                 6,448   6,080
  //   MD5, 256 MiB (without the padding block)
  //     262,144            1,376 (825)     1,382 (833)
  //     1,048,576          1,405 (845)     1,383 (833)
  //     67,108,864         1,879 (1,850)   1,570 (1,560)
  if (sig != kSigDjb2) return n_keys > (1ull << 19) ? kFragMostKeys : kFragFewKeys;
  return n_keys > (1ull << 22) ? kFragMostKeys : n_keys > (1ull << 18) ? kFragManyKeys : kFragFewKeys;
}

uint64_t frag_windows(uint64_t n_bytes) { return n_bytes >= 64 ? (n_bytes - 64) / kFragStride + 1 : 0; }

uint64_t frag_tiles(int sig, uint64_t n_bytes) {
  Geom g;
  if (!geom(sig, kLayoutHash, kFragFewKeys, false, &g)) return 0;
  return (frag_windows(n_bytes) + g.tile_win - 1) / g.tile_win;
}

bool frag_sig_supported(int sig) { return sig == kSigMd5 || sig == kSigMd5NoPad || sig == kSigDjb2; }

int frag_digests(int sig, const uint8_t* arena, uint64_t n, uint4* dig, uint8_t* trivial, int sms, void* stream) {
  if (!n) return 0;
  const unsigned g = (unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)sms * 8);
  cudaStream_t st = (cudaStream_t)stream;
  if (sig == kSigMd5) frag_digest_kernel<kSigMd5><<<g, 256, 0, st>>>(arena, n, dig, trivial, 1u);
  else if (sig == kSigMd5NoPad) frag_digest_kernel<kSigMd5NoPad><<<g, 256, 0, st>>>(arena, n, dig, trivial, 1u);
  else if (sig == kSigDjb2) frag_digest_kernel<kSigDjb2><<<g, 256, 0, st>>>(arena, n, dig, trivial, 1u);
  else return (int)cudaErrorInvalidValue;
  return (int)cudaGetLastError();
}

int frag_bloom(int sig, const uint4* slots, uint32_t n_slots, uint64_t n_keys, uint32_t* words, uint32_t mask,
               uint32_t* l1, int sms, void* stream) {
  const unsigned g = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(((uint64_t)n_slots + 255) / 256, (uint64_t)sms * 8));
  const int keys = frag_key_class(sig, n_keys);
  void (*fn)(const uint4*, uint32_t, uint32_t*, uint32_t, uint32_t*);
  if (sig == kSigDjb2)
    fn = keys == kFragMostKeys   ? frag_bloom_kernel<kSigDjb2, kFragMostKeys>
         : keys == kFragManyKeys ? frag_bloom_kernel<kSigDjb2, kFragManyKeys>
                                 : frag_bloom_kernel<kSigDjb2, kFragFewKeys>;
  else
    fn = keys == kFragMostKeys ? frag_bloom_kernel<kSigMd5, kFragMostKeys> : frag_bloom_kernel<kSigMd5, kFragFewKeys>;
  fn<<<g, 256, 0, (cudaStream_t)stream>>>(slots, n_slots, words, mask, l1);
  return (int)cudaGetLastError();
}

int frag_window_sigs(int sig, const uint8_t* image, uint64_t n_bytes, uint4* out, int sms, void* stream) {
  const uint64_t n_win = frag_windows(n_bytes);
  if (!n_win) return 0;
  const void* fn;
  uint32_t win, bytes;
  switch (sig) {
    case kSigMd5:
      fn = (const void*)frag_window_sig_kernel<kSigMd5>;
      win = FragSigTile<kSigMd5>::kWin;
      bytes = FragSigTile<kSigMd5>::kBytes;
      break;
    case kSigMd5NoPad:
      fn = (const void*)frag_window_sig_kernel<kSigMd5NoPad>;
      win = FragSigTile<kSigMd5NoPad>::kWin;
      bytes = FragSigTile<kSigMd5NoPad>::kBytes;
      break;
    case kSigDjb2:
      fn = (const void*)frag_window_sig_kernel<kSigDjb2>;
      win = FragSigTile<kSigDjb2>::kWin;
      bytes = FragSigTile<kSigDjb2>::kBytes;
      break;
    default: return (int)cudaErrorInvalidValue;
  }
  const uint64_t tiles = (n_win + win - 1) / win;
  const uint32_t smem = 8 * bytes;  // 8 warps of 256 threads
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return (int)e;
  const unsigned grid = (unsigned)std::min<uint64_t>((tiles + 7) / 8, (uint64_t)sms * 8);
  uint32_t one = 1u;
  void* args[] = {&image, &n_bytes, (void*)&n_win, (void*)&tiles, &out, &one};
  return (int)cudaLaunchKernel(fn, dim3(grid), dim3(256), args, smem, (cudaStream_t)stream);
}

FragImages frag_images(const FragImage* host, const FragImage* dev, size_t n) {
  FragImages l;
  memset(&l, 0, sizeof l);
  l.dev = dev;
  l.n = (uint32_t)n;
  for (size_t k = 0; k < n && n <= kInlineSegs; k++) l.in[k] = host[k];
  return l;
}

int frag_count(const TableView& tab, const FragImages& images, uint64_t n_tiles, uint64_t* tile_ntrip, const FragHits& hits,
               uint32_t* status, unsigned long long* rejected, int sms, void* stream) {
  FragParams p = make_params(tab, images, n_tiles, hits, status);
  p.rejected = rejected;
  if (!p.n_tiles) return 0;
  const bool multi = images.n > 1;
  FragDev* d;
  int rc = frag_device(&d);
  if (rc) return rc;
  Geom g;
  const int keys = frag_key_class((int)tab.sig, tab.n_keys);
  if (!geom((int)tab.sig, tab.layout, keys, multi, &g)) return (int)cudaErrorInvalidValue;
  if (tab.sig == kSigDjb2 && !tab.frag_l1) return (int)cudaErrorInvalidValue;  // the kernel copies it in
  p.tile_ntrip = tile_ntrip;
  const uint64_t cap =
      tab.sig == kSigDjb2 ? (uint64_t)sms * (uint64_t)d->count_blocks[tab.sig][tab.layout][keys][multi] : INT32_MAX;
  const uint64_t warps_per_block = (uint64_t)g.threads / 32;
  const unsigned grid = (unsigned)std::min<uint64_t>((p.n_tiles + warps_per_block - 1) / warps_per_block, cap);
  void* args[] = {&p};
  return (int)cudaLaunchKernel(g.count, dim3(grid), dim3(g.threads), args, g.smem_count, (cudaStream_t)stream);
}

int frag_emit(const TableView& tab, const FragImages& images, uint64_t n_tiles, const uint64_t* tile_off,
              const uint64_t* total, const FragHits& hits, MatchOut* out, uint64_t out_cap, uint32_t* status, int sms,
              void* stream) {
  FragParams p = make_params(tab, images, n_tiles, hits, status);
  if (!p.n_tiles) return 0;
  Geom g;
  if (!geom((int)tab.sig, tab.layout, kFragFewKeys, false, &g)) return (int)cudaErrorInvalidValue;
  p.tile_off = tile_off;
  p.total = total;
  p.out = out;
  p.out_cap = out_cap;
  const uint64_t warps_per_block = kEmitThreads / 32;
  const unsigned grid = (unsigned)std::min<uint64_t>((p.n_tiles + warps_per_block - 1) / warps_per_block,
                                                     (uint64_t)sms * 8);
  void* args[] = {&p};
  return (int)cudaLaunchKernel(g.emit, dim3(grid), dim3(kEmitThreads), args, 0, (cudaStream_t)stream);
}

}  // namespace cvk
