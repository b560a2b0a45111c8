// Device kernels that build the master signature table (paper Section 3.1: every master
// sector's signature is inserted at the slot given by its low bits, collisions resolved by
// linear probing, Eq. 3).
//
// Steps (one launch each):
//   postings the (file_id, file_sector) of every master sector, in master order.
//   insert   one thread per master sector: claim the first free slot from the digest's home
//            slot on (atomicCAS of its owner word), or join the slot that already holds an equal
//            digest; record the slot, track the longest probe run.
//   slots    an exclusive scan of the member counts gives every key its postings; one pass over the
//            slots writes their records, the postings of keys with one member and the Bloom
//            filter's bits.
//   members  (only for keys with several members) these members, in master order, are sorted by
//            their key's first posting (stable LSD radix sort) and take the postings from there
//            on, so they are in master order, i.e. by (file_id, file_sector).
//   sorted   (sorted layout only) the occupied slots, compacted in slot order, are sorted by
//            h0 and become the searched array.
// Position-keyed tables (one S_tau per cluster position, Section 3.1) key every slot by
// (digest, tau) with tau = file_sector mod 8; the steps are the same.
// Which slot a digest lands in depends on thread timing; the lookup result does not.
#pragma once
#include <stdint.h>

#include "cv_internal.h"

namespace cvk {

// Posting of every master sector: its file, by binary search of file_base (n_files + 1 entries:
// first master index of every file, then the total), and its sector in the file. With tau (position-
// keyed tables), tau[m] = file_sector mod 8.
// A warp takes kPostRun consecutive sectors: two searches over all files for its first and last one,
// then short ones between them.
constexpr uint32_t kPostRun = 512;

__device__ __forceinline__ uint32_t file_of(const uint64_t* file_base, uint32_t lo, uint32_t hi, uint64_t m) {
  while (hi - lo > 1) {  // largest f in [lo, hi) with file_base[f] <= m
    const uint32_t mid = (lo + hi) >> 1;
    if (file_base[mid] <= m) lo = mid; else hi = mid;
  }
  return lo;
}

__global__ void unit_postings_kernel(const uint64_t* file_base, uint32_t n_files, uint64_t n, uint2* post,
                                     uint8_t* tau) {
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  for (uint64_t m0 = ((uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kPostRun; m0 < n;
       m0 += warps * kPostRun) {
    const uint64_t end = m0 + kPostRun < n ? m0 + kPostRun : n;
    const uint32_t f0 = file_of(file_base, 0, n_files, m0), f1 = file_of(file_base, f0, n_files, end - 1) + 1;
    for (uint64_t m = m0 + (threadIdx.x & 31); m < end; m += 32) {
      const uint32_t f = file_of(file_base, f0, f1, m);
      const uint32_t s = (uint32_t)(m - file_base[f]);
      post[m] = make_uint2(f, s);
      if (tau) tau[m] = (uint8_t)(s & 7u);
    }
  }
}

// tau: per master sector position (position-keyed tables), or null for one table over all
// positions (every tau 0). The key is (digest, tau). A slot's owner is the master index of its key's
// first member + 1 (0: empty), its extra the number of other members. Bound by the latency of
// the random accesses (owner and count in one 8-byte word took 248 us against 178 for 4,194,304 keys,
// and 333 us with a second atomic that counts every member).
// (Claiming slots from the kernel that hashes the sectors saved nothing: waited for at once, the
// atomics held up the hashing by 220 us; looked at a tile later, by 100, and the keys whose home was
// taken still took 153.)
__global__ void insert_kernel(const uint4* dig, const uint8_t* trivial, const uint8_t* tau, uint64_t n,
                              uint32_t* owner, uint32_t* extra, uint32_t* slot_of, uint32_t mask, uint32_t* max_disp,
                              uint32_t* n_kept, uint32_t* status) {
  const uint32_t none = mask + 1u;
  uint32_t kept = 0, longest = 0;  // this thread's, added to the shared counters once per warp
  for (uint64_t m = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (uint64_t)gridDim.x * blockDim.x) {
    if (trivial[m]) {
      slot_of[m] = none;
      continue;
    }
    const uint4 d = dig[m];
    const uint32_t t = tau ? tau[m] : 0u;
    uint32_t idx = tau_home(d.x, t) & mask;
    uint32_t c = 0;
    bool placed = false;
    for (; c <= mask; c++) {
      const uint32_t prev = atomicCAS(owner + idx, 0u, (uint32_t)m + 1u);
      if (prev == 0u) {
        placed = true;
        break;
      }
      const uint4 e = dig[prev - 1u];
      const uint32_t te = tau ? tau[prev - 1u] : 0u;
      if (e.x == d.x && e.y == d.y && e.z == d.z && e.w == d.w && te == t) {
        atomicAdd(extra + idx, 1u);
        placed = true;
        break;
      }
      idx = (idx + 1u) & mask;
    }
    if (!placed) {
      atomicOr(status, kStTableFull);
      slot_of[m] = none;
      continue;
    }
    slot_of[m] = idx;
    longest = c > longest ? c : longest;
    kept++;
  }
  // one update per warp: a per-key atomic on one address serialises the whole build
  kept = __reduce_add_sync(0xFFFFFFFFu, kept);
  longest = __reduce_max_sync(0xFFFFFFFFu, longest);
  if ((threadIdx.x & 31) == 0 && kept) {
    atomicAdd(n_kept, kept);
    atomicMax(max_disp, longest);
  }
}

// The same for many keys and at most half of the slots taken. What costs time above is that a thread
// has one atomic in flight and a warp waits for its longest walk each time. Here a thread's six units
// try their home slots together, and those that find an owner there are gathered in shared memory and
// taken one per thread, each walking on by itself. Neighbours with one home slot (copies of a sector)
// let the first of them try, and lanes that find themselves with one key count as one, or they would
// queue at one address (a build of 4,194,304 sectors, two alternating: 2,760 us with an addition for each
// copy, 2,238 so, 2,657 by the sort that was before; of 2^20 equal ones 1,060 and 407). Both kernels, us:
//   keys         load      one by one   here (4, 6, 12 units a thread)
//   100,000      38%       13           18, 24, 31
//   300,000      29%       18           15, 16, 25
//   1,048,576    25%       42           21, 22, 28
//   1,900,000    45%       65           49, 55, 60
//   4,194,304    25%       178          120, 109, 101
//   7,600,000    45%       327          258, 237, 266
//   900,000      86%       290          425, 345, 420
//   7,000,000    83%       1,140        768, 800, 830
// so it is used from 2^18 keys on, and where walks are long, above half, not at all (the few longest
// walks decide there, and the more keys are under way at once the longer they get).
constexpr uint64_t kInsertChunksMin = 1ull << 18;
constexpr int kInsertThreads = 128;
constexpr int kInsertUnits = 6;   // per thread
constexpr uint32_t kInsertChunk = kInsertThreads * kInsertUnits;

__global__ void __launch_bounds__(kInsertThreads, 10)
    insert_chunks_kernel(const uint4* dig, const uint8_t* trivial, const uint8_t* tau, uint64_t n, uint32_t* owner,
                  uint32_t* extra, uint32_t* slot_of, uint32_t mask, uint32_t* max_disp, uint32_t* n_kept,
                  uint32_t* status) {
  __shared__ uint2 s_taken[kInsertChunk];  // units whose home slot has an owner: the unit, that owner
  __shared__ uint32_t s_n, s_kept, s_longest;
  const uint32_t none = mask + 1u;
  const uint64_t c0 = (uint64_t)blockIdx.x * kInsertChunk + threadIdx.x;
  const uint32_t lane = threadIdx.x & 31;
  uint32_t kept = 0, longest = 0;
  if (threadIdx.x == 0) s_n = s_kept = s_longest = 0;
  uint32_t home[kInsertUnits], held[kInsertUnits];
  bool live[kInsertUnits];
#pragma unroll
  for (int u = 0; u < kInsertUnits; u++) {
    const uint64_t m = c0 + u * kInsertThreads;
    live[u] = m < n && !trivial[m];
    if (m < n && !live[u]) slot_of[m] = none;
    home[u] = live[u] ? tau_home(dig[m].x, tau ? tau[m] : 0u) & mask : none;
  }
  __syncthreads();
  // of neighbours with one home slot the first tries for all of them
  uint32_t heads[kInsertUnits];
#pragma unroll
  for (int u = 0; u < kInsertUnits; u++) {
    const uint32_t before = __shfl_up_sync(0xFFFFFFFFu, home[u], 1);
    const bool head = lane == 0u || home[u] != before;
    heads[u] = __ballot_sync(0xFFFFFFFFu, head);
    held[u] = live[u] && head ? atomicCAS(owner + home[u], 0u, (uint32_t)(c0 + u * kInsertThreads) + 1u) : 0u;
  }
#pragma unroll
  for (int u = 0; u < kInsertUnits; u++) {
    const uint32_t m = (uint32_t)(c0 + u * kInsertThreads);
    const uint32_t from = 31u - __clz(heads[u] << (31u - lane) >> (31u - lane));
    const uint32_t by = __shfl_sync(0xFFFFFFFFu, held[u] ? held[u] : m + 1u, from);
    if (from != lane) held[u] = by;
  }
#pragma unroll
  for (int u = 0; u < kInsertUnits; u++) {
    if (!live[u]) continue;
    const uint32_t m = (uint32_t)(c0 + u * kInsertThreads);
    if (held[u] == 0u) {
      slot_of[m] = home[u];
      kept++;
    } else {
      s_taken[atomicAdd(&s_n, 1u)] = make_uint2(m, held[u]);
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < s_n; i += kInsertThreads) {
    const uint32_t m = s_taken[i].x;
    const uint4 d = dig[m];
    const uint32_t t = tau ? tau[m] : 0u;
    uint32_t idx = tau_home(d.x, t) & mask, c = 0, by = s_taken[i].y;
    while (by) {  // the slot has an owner: this key's, or the next slot is tried
      const uint4 e = dig[by - 1u];
      const uint32_t te = tau ? tau[by - 1u] : 0u;
      if (e.x == d.x && e.y == d.y && e.z == d.z && e.w == d.w && te == t) {
        // one addition for the lanes that are here with one key
        const uint32_t peers = __match_any_sync(__activemask(), idx);
        if ((peers & ((1u << lane) - 1u)) == 0u) atomicAdd(extra + idx, __popc(peers));
        break;
      }
      if (c == mask) {
        atomicOr(status, kStTableFull);
        idx = none;
        break;
      }
      idx = (idx + 1u) & mask;
      c++;
      by = atomicCAS(owner + idx, 0u, m + 1u);
    }
    slot_of[m] = idx;
    if (idx == none) continue;
    longest = c > longest ? c : longest;
    kept++;
  }
  // one update per block: a per-key atomic on one address serialises the whole build
  kept = __reduce_add_sync(0xFFFFFFFFu, kept);
  longest = __reduce_max_sync(0xFFFFFFFFu, longest);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&s_kept, kept);
    atomicMax(&s_longest, longest);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_kept) atomicAdd(n_kept, s_kept);
    if (s_longest) atomicMax(max_disp, s_longest);
  }
}

// ------------------------------------------------------------------ stable radix sort pass
constexpr int kRsThreads = 256;
constexpr int kRsRounds = 16;
constexpr int kRsChunk = kRsThreads * kRsRounds;

// Digit histogram of each 4096-key chunk: hist[digit * n_blocks + block].
__global__ void __launch_bounds__(kRsThreads) rs_hist_kernel(const uint32_t* keys, uint64_t n, int shift,
                                                             uint32_t* hist, uint32_t n_blocks) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const uint64_t base = (uint64_t)blockIdx.x * kRsChunk;
  for (int r = 0; r < kRsRounds; r++) {
    const uint64_t i = base + (uint64_t)r * kRsThreads + threadIdx.x;
    if (i < n) atomicAdd(h + ((keys[i] >> shift) & 255u), 1u);
  }
  __syncthreads();
  hist[(uint64_t)threadIdx.x * n_blocks + blockIdx.x] = h[threadIdx.x];
}

// In-place exclusive scan of n u32 values whose total fits in 32 bits, over the whole GPU in
// three launches: the sum of every 4096-value chunk; an exclusive scan of those sums (one
// block); each chunk's own scan, offset by its sum's prefix. Loads and stores are coalesced;
// the per-thread runs are read from a padded shared tile without bank conflicts.
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr uint32_t kScanChunk = kScanThreads * kScanItems;

// Exclusive scan of x over the B threads of a block; *total gets the sum (every thread).
template <int B>
__device__ __forceinline__ uint32_t block_exclusive_u32(uint32_t x, uint32_t* total) {
  __shared__ uint32_t ws[B / 32 + 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= d) incl += y;
  }
  if (lane == 31) ws[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = lane < B / 32 ? ws[lane] : 0u;
    uint32_t wi = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, wi, d);
      if (lane >= d) wi += y;
    }
    if (lane < B / 32) ws[lane] = wi - w;
    if (lane == B / 32 - 1) ws[B / 32] = wi;
  }
  __syncthreads();
  const uint32_t r = ws[warp] + incl - x;
  *total = ws[B / 32];
  __syncthreads();  // ws may be reused by the next call
  return r;
}

__global__ void __launch_bounds__(kScanThreads) scan_chunk_sums_u32_kernel(const uint32_t* v, uint64_t n,
                                                                           uint32_t* sums) {
  const uint64_t base = (uint64_t)blockIdx.x * kScanChunk;
  uint32_t s = 0;
#pragma unroll
  for (int r = 0; r < kScanItems; r++) {
    const uint64_t i = base + (uint64_t)r * kScanThreads + threadIdx.x;
    if (i < n) s += v[i];
  }
  uint32_t total;
  block_exclusive_u32<kScanThreads>(s, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) scan_sums_u32_kernel(uint32_t* sums, uint32_t nb) {
  uint32_t carry = 0;
  for (uint32_t t0 = 0; t0 < nb; t0 += 1024) {
    const uint32_t i = t0 + threadIdx.x;
    const uint32_t x = i < nb ? sums[i] : 0u;
    uint32_t total;
    const uint32_t e = block_exclusive_u32<1024>(x, &total);
    if (i < nb) sums[i] = carry + e;
    carry += total;
  }
}

__global__ void __launch_bounds__(kScanThreads) scan_chunks_u32_kernel(uint32_t* v, uint64_t n, const uint32_t* sums) {
  __shared__ uint32_t tile[kScanChunk + kScanChunk / 32];  // element e at e + e / 32
  const uint64_t base = (uint64_t)blockIdx.x * kScanChunk;
  const int tid = threadIdx.x;
#pragma unroll
  for (int r = 0; r < kScanItems; r++) {
    const uint32_t e = r * kScanThreads + tid;
    const uint64_t i = base + e;
    tile[e + e / 32] = i < n ? v[i] : 0u;
  }
  __syncthreads();
  uint32_t loc[kScanItems];
  uint32_t s = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; j++) {
    const uint32_t e = tid * kScanItems + j;
    loc[j] = tile[e + e / 32];
    s += loc[j];
  }
  uint32_t total;
  uint32_t run = block_exclusive_u32<kScanThreads>(s, &total) + sums[blockIdx.x];
#pragma unroll
  for (int j = 0; j < kScanItems; j++) {
    const uint32_t e = tid * kScanItems + j;
    tile[e + e / 32] = run;
    run += loc[j];
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kScanItems; r++) {
    const uint32_t e = r * kScanThreads + tid;
    const uint64_t i = base + e;
    if (i < n) v[i] = tile[e + e / 32];
  }
}

// Scatter of one pass: the keys of a chunk go, in their original order within each digit, to
// the chunk's offset for that digit (hist, after the scan).
__global__ void __launch_bounds__(kRsThreads) rs_scatter_kernel(const uint32_t* kin, const uint32_t* vin,
                                                                uint32_t* kout, uint32_t* vout, uint64_t n, int shift,
                                                                const uint32_t* hist, uint32_t n_blocks) {
  constexpr int kWarps = kRsThreads / 32;
  __shared__ uint32_t run[256];
  __shared__ uint32_t wcnt[kWarps][256];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lane_lt = (1u << lane) - 1u;
  run[tid] = hist[(uint64_t)tid * n_blocks + blockIdx.x];
  const uint64_t base = (uint64_t)blockIdx.x * kRsChunk;
  for (int r = 0; r < kRsRounds; r++) {
#pragma unroll
    for (int w = 0; w < kWarps; w++) wcnt[w][tid] = 0;
    __syncthreads();
    const uint64_t i = base + (uint64_t)r * kRsThreads + tid;
    const bool valid = i < n;
    const uint32_t key = valid ? kin[i] : 0u;
    const uint32_t digit = valid ? ((key >> shift) & 255u) : 256u;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, digit);
    const uint32_t rank = __popc(peers & lane_lt);
    if (valid && rank == 0) wcnt[warp][digit] = __popc(peers);
    __syncthreads();
    if (valid) {
      uint32_t pos = run[digit] + rank;
      for (int w = 0; w < warp; w++) pos += wcnt[w][digit];
      kout[pos] = key;
      vout[pos] = vin[i];
    }
    __syncthreads();
    uint32_t tot = 0;
#pragma unroll
    for (int w = 0; w < kWarps; w++) tot += wcnt[w][tid];
    run[tid] += tot;
    __syncthreads();
  }
}

// ------------------------------------------------------------------------------ slots
// The slots in chunks of kSlotChunk, a block each; a warp has 128 consecutive slots, in four rows of
// 32. first[c] holds the members of the chunks before chunk c: the chunks' sums, read in a pass of
// their own (8 bytes a slot) and scanned. With decoupled look-back instead, in one pass, the kernel took
// 400 us for the same table: some 300 chunks are under way at a time, none of them with an
// inclusive prefix yet, and each walked back over all of them.
//
// Bound by memory: 8 bytes read and 32 written per slot (4,194,304 keys in 2^24 slots: 671 MB),
// two random sectors read per key, a Bloom block updated per key. A slot record is one 32-byte store.
// Of a key's eight Bloom bits eight lanes each set one, so that the block is one update in L2. This
// takes 204 us and the sums 25, where sorting (slot, master) pairs, filling postings and slots, a pass
// for the Bloom filter and clearing the slots and counts took 804.
constexpr int kSlotThreads = 256;
constexpr int kSlotRows = 4;
constexpr uint32_t kSlotChunk = kSlotThreads * kSlotRows;

// sums[c] = members of the keys in chunk c.
__global__ void __launch_bounds__(kSlotThreads) slot_sums_kernel(const uint32_t* owner, const uint32_t* extra, uint32_t n_slots,
                                                                 uint32_t* sums) {
  const uint64_t base = (uint64_t)blockIdx.x * kSlotChunk + threadIdx.x;
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kSlotRows; k++) {
    const uint64_t i = base + (uint64_t)k * kSlotThreads;
    if (i < n_slots) s += extra[i] + (owner[i] ? 1u : 0u);
  }
  uint32_t total;
  block_exclusive_u32<kSlotThreads>(s, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Evicted first, like the owners that have been read: the digests and postings that the slots gather
// stay in L2 for longer (215 to 204 us for 16.8M slots).
__device__ __forceinline__ void store_slot(uint4* p, uint4 a, uint4 b) {
  asm volatile("st.global.L2::evict_first.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z),
               "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}

// counters: [0] keys, [1] members of keys with several. post: posting per master index; member: the
// master index of every posting (null: not wanted). tags: a byte per slot (null: not wanted). bloom: null
// for none.
__global__ void __launch_bounds__(kSlotThreads) table_slots_kernel(
    const uint32_t* owners, const uint32_t* extra, uint32_t n_slots, const uint32_t* first, const uint4* dig, const uint8_t* tau,
    const uint2* post, uint4* slots, uint8_t* tags, uint2* postings, uint32_t* member, uint32_t* bloom, uint32_t bloom_mask,
    uint32_t* counters) {
  constexpr int kWarps = kSlotThreads / 32;
  constexpr uint32_t kFull = 0xFFFFFFFFu;
  __shared__ uint32_t s_warp[kWarps];
  __shared__ uint32_t s_key[kWarps][32 * kSlotRows][3];  // d1, d2, Bloom block of the warp's keys
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t base = (uint64_t)blockIdx.x * kSlotChunk + warp * 32u * kSlotRows + lane;
  uint32_t owner[kSlotRows], cnt[kSlotRows], before[kSlotRows], t[kSlotRows];
  uint4 d[kSlotRows];
  uint2 po[kSlotRows];
#pragma unroll
  for (int k = 0; k < kSlotRows; k++) {
    const bool in = base + 32u * k < n_slots;
    owner[k] = in ? __ldcs(owners + base + 32u * k) : 0u;
    cnt[k] = in ? __ldcs(extra + base + 32u * k) + (owner[k] ? 1u : 0u) : 0u;
  }
#pragma unroll
  for (int k = 0; k < kSlotRows; k++) {
    d[k] = owner[k] ? dig[owner[k] - 1u] : make_uint4(0, 0, 0, 0);
    po[k] = owner[k] ? post[owner[k] - 1u] : make_uint2(0, 0);
    t[k] = owner[k] && tau ? tau[owner[k] - 1u] : 0u;
  }
  // exclusive scan of the counts within the warp's slots, then over the warps
  uint32_t sum = 0, keys = 0, several = 0;
#pragma unroll
  for (int k = 0; k < kSlotRows; k++) {
    uint32_t incl = cnt[k];
#pragma unroll
    for (int q = 1; q < 32; q <<= 1) {
      const uint32_t v = __shfl_up_sync(kFull, incl, q);
      if (lane >= (uint32_t)q) incl += v;
    }
    before[k] = sum + incl - cnt[k];
    sum += __shfl_sync(kFull, incl, 31);
    several += cnt[k] > 1u ? cnt[k] : 0u;
  }
  if (lane == 0) s_warp[warp] = sum;
  __syncthreads();
  uint32_t off0 = first[blockIdx.x];
  for (uint32_t w = 0; w < warp; w++) off0 += s_warp[w];
#pragma unroll
  for (int k = 0; k < kSlotRows; k++) {
    const uint64_t i = base + 32u * k;
    const uint32_t off = off0 + before[k];
    const uint32_t has = __ballot_sync(kFull, owner[k] != 0u);
    if (tags && i < n_slots) tags[i] = cnt[k] ? (uint8_t)slot_tag(d[k].z) : 0;
    if (i < n_slots) store_slot(slots + 2 * i, d[k], make_uint4(owner[k] ? off : 0u, cnt[k], t[k], 0u));
    if (cnt[k] == 1u) {
      postings[off] = po[k];
      if (member) member[off] = owner[k] - 1u;
    }
    if (bloom && owner[k]) {
      uint32_t* e = s_key[warp][keys + __popc(has & ((1u << lane) - 1u))];
      e[0] = d[k].y;
      e[1] = d[k].z;
      e[2] = tau_block(d[k].w, t[k]) & bloom_mask;
    }
    keys += __popc(has);
  }
  if (bloom) {
    __syncwarp();
    const uint32_t word = lane & 7u;  // the Bloom bit in word j: d1 >> 5j for j < 6, d2 >> 5(j - 6) else
    for (uint32_t e = lane >> 3; e < keys; e += 4) {
      const uint32_t* key = s_key[warp][e];
      const uint32_t b = word < 6u ? key[0] >> (5u * word) : key[1] >> (5u * (word - 6u));
      atomicOr(bloom + 8ull * key[2] + word, 1u << (b & 31u));
    }
  }
  several = __reduce_add_sync(kFull, several);
  __shared__ uint32_t s_keys, s_several;
  if (threadIdx.x == 0) s_keys = s_several = 0;
  __syncthreads();
  if (lane == 0 && keys) {
    atomicAdd(&s_keys, keys);
    if (several) atomicAdd(&s_several, several);
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_keys) {  // one update per block
    atomicAdd(counters, s_keys);
    if (s_several) atomicAdd(counters + 1, s_several);
  }
}

// ---------------------------------------------------------------------------- members
// 1 for every master unit whose key has several members, else 0.
__global__ void several_flags_kernel(const uint32_t* slot_of, uint64_t n, uint32_t n_slots, const uint32_t* extra,
                                     uint32_t* flags) {
  for (uint64_t m = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (uint64_t)gridDim.x * blockDim.x)
    flags[m] = slot_of[m] < n_slots && extra[slot_of[m]] > 0u ? 1u : 0u;
}

// These units in master order (at: the exclusive scan of the flags), keyed by their key's first posting.
__global__ void several_keys_kernel(const uint32_t* slot_of, uint64_t n, uint32_t n_slots, const uint4* slots,
                                    const uint32_t* at, uint32_t* keys, uint32_t* vals) {
  for (uint64_t m = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; m < n; m += (uint64_t)gridDim.x * blockDim.x) {
    if (slot_of[m] >= n_slots) continue;
    const uint4 val = slots[2ull * slot_of[m] + 1];
    if (val.y <= 1u) continue;
    keys[at[m]] = val.x;
    vals[at[m]] = (uint32_t)m;
  }
}

// Sorted by key: the members of a key take its postings in this order.
__global__ void several_postings_kernel(const uint32_t* keys, const uint32_t* vals, uint32_t n, const uint2* post,
                                        uint2* postings, uint32_t* member) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t key = keys[i];
    uint32_t lo = 0, hi = i;  // the key's first place
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (keys[mid] < key) lo = mid + 1; else hi = mid;
    }
    postings[key + i - lo] = post[vals[i]];
    if (member) member[key + i - lo] = vals[i];
  }
}

// Kept master units (sectors or fragments of wpu 16-byte words) in posting order: posting q is
// master unit member[q]; its words go to out + wpu q. One thread per 16-byte word.
__global__ void gather_units_kernel(const uint4* arena, const uint32_t* member, uint64_t n, uint32_t wpu, uint4* out) {
  const uint64_t words = n * wpu;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = arena[(uint64_t)member[i / wpu] * wpu + i % wpu];
}

// ------------------------------------------------------------------- sorted layout
// Sort key of the occupied-slot compaction: 0 for an occupied slot, 1 for an empty one; a stable
// sort by it puts the occupied slots first, in slot order.
__global__ void occupied_keys_kernel(const uint4* slots, uint32_t n_slots, uint32_t* keys, uint32_t* vals) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_slots; i += gridDim.x * blockDim.x) {
    keys[i] = slots[2ull * i + 1].y != 0u ? 0u : 1u;
    vals[i] = i;
  }
}

// h0 = tau_home(d0, tau) of the slots vals[0..n).
__global__ void h0_keys_kernel(const uint4* slots, const uint32_t* vals, uint32_t n, uint32_t* keys) {
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const uint32_t i = vals[q];
    keys[q] = tau_home(slots[2ull * i].x, slots[2ull * i + 1].z);
  }
}

// Slot records in the order of vals (ascending h0): out[q] = slots[vals[q]].
__global__ void gather_slots_kernel(const uint4* slots, const uint32_t* vals, uint32_t n, uint4* out) {
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const uint32_t i = vals[q];
    out[2ull * q] = slots[2ull * i];
    out[2ull * q + 1] = slots[2ull * i + 1];
  }
}

// The index over the sorted keys: start[b] = the first key whose top bits are b or more, a search
// per bucket.
__global__ void key_index_kernel(const uint32_t* keys, uint32_t n, uint32_t shift, uint32_t* start) {
  const uint64_t buckets = 1ull << (32 - shift);
  for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= buckets;
       b += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
      const uint32_t mid = lo + (hi - lo) / 2;
      if ((uint64_t)keys[mid] < (b << shift)) lo = mid + 1; else hi = mid;
    }
    start[b] = lo;
  }
}

// ------------------------------------------------------------------- loaded tables
// Every occupied record of a loaded table must name postings inside [0, n_postings).
__global__ void validate_slots_kernel(const uint4* slots, uint64_t n, uint64_t n_postings, uint32_t* status) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint4 val = slots[2 * i + 1];
    if (val.y != 0u && (uint64_t)val.x + val.y > n_postings) atomicOr(status, kStBadTable);
  }
}

// The tags of a loaded table's slots.
__global__ void slot_tags_kernel(const uint4* slots, uint64_t n, uint8_t* tags) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    tags[i] = slots[2 * i + 1].y ? (uint8_t)slot_tag(slots[2 * i].z) : 0;
}

// ----------------------------------------------------------------------------- Bloom
__global__ void bloom_kernel(const uint4* slots, uint32_t n_slots, uint32_t* bloom, uint32_t bloom_mask) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_slots; i += gridDim.x * blockDim.x) {
    const uint4 val = slots[2ull * i + 1];
    if (val.y == 0u) continue;
    const uint4 d = slots[2ull * i];
    uint32_t* blk = bloom + 8ull * (tau_block(d.w, val.z) & bloom_mask);
    atomicOr(blk + 0, 1u << (d.y & 31));
    atomicOr(blk + 1, 1u << ((d.y >> 5) & 31));
    atomicOr(blk + 2, 1u << ((d.y >> 10) & 31));
    atomicOr(blk + 3, 1u << ((d.y >> 15) & 31));
    atomicOr(blk + 4, 1u << ((d.y >> 20) & 31));
    atomicOr(blk + 5, 1u << ((d.y >> 25) & 31));
    atomicOr(blk + 6, 1u << (d.z & 31));
    atomicOr(blk + 7, 1u << ((d.z >> 5) & 31));
  }
}

}  // namespace cvk
