// Second half of the match compaction: the per-tile triple counts of the scan are turned into
// output offsets by one exclusive scan, then every hit record of every tile is expanded into
// its (disk_sector, file_id, file_sector) triples, in one kernel for scans of up to kFinishTiles
// output tiles and in three for larger ones. Tiles are in sector order, the records of a
// tile are in sector order (ballot ranks), and each digest's postings are sorted by
// (file_id, file_sector), so the output is sorted without a sort; the only waits between thread
// blocks are the offset scan's bounded look-back. (The paper's Section 3.2 writes matches to a
// host-visible buffer in no stated order; the sorted triple list is this library's output
// format.)
#pragma once
#include <stdint.h>

#include "cv_internal.h"

namespace cvk {

// Exclusive scan of the per-tile triple counts in one pass: each block scans a chunk and adds
// its predecessors' published sums (decoupled look-back, every wait bounded). A second small pass
// reads off each segment's first offset. (The kernels are in kernels_scan.cu; this header holds
// the expand pass, instantiated with each configuration.)
constexpr int kOffThreads = 1024;
constexpr int kOffItems = 4;
constexpr uint64_t kOffChunk = (uint64_t)kOffThreads * kOffItems;

// What the passes after a scan read and write.
struct CompactParams {
  const uint4* hit_rec;        // the scan's outputs
  const uint32_t* tile_nhit;
  const uint64_t* tile_ntrip;
  uint64_t n_out_tiles;
  SegList segs;
  const uint2* postings;
  const uint8_t* confirm;      // 64-bit signatures: the postings' master sectors, else null
  MatchOut* out;
  uint64_t out_cap;
  uint32_t* status;
  const uint64_t* tile_off;    // expand pass: output offset per tile
  uint64_t* seg_off;           // one-kernel pass: out, the offset of every segment's first tile
  uint64_t* total;             // out, the sum of the triple counts
  unsigned long long* nhit_sum;  // the sectors with a match are added to it (null: not counted)
};

// A warp takes 32 consecutive output tiles (32 sectors each) at a time: lane b describes tile
// u0 + b, my_n records that begin at output offset my_off. A hit record is {lane, post_off, post_cnt,
// n_emit}: the sector emits n_emit triples, all of its postings, or with a 64-bit signature
// (confirm != null) those whose master sector equals the disk sector byte for byte (compared again
// only if some did not: comparing always took 31 us instead of 9 on a 2 GiB CRC64 image). The
// records of the group's tiles with hits are numbered in tile order and taken 32 at a time, one per
// lane, so that the dependent loads of different tiles (record, posting) are in flight together:
// most tiles have no hit, and a tile's few hits would otherwise each wait in turn. A record's place
// in the output is its tile's offset plus the triples of the records before it in the tile (a
// segmented warp scan, carried across passes). out_cap bounds the writes (kStOverflow when exceeded).
template <int T>
__device__ __forceinline__ void expand_group(const CompactParams& p, uint64_t u0, uint32_t my_n, uint32_t my_first,
                                             uint32_t n_rec, uint64_t my_off) {
  constexpr uint32_t kW = T / 32;
  constexpr uint32_t kFull = 0xFFFFFFFFu;
  const uint32_t lane = threadIdx.x & 31;
  // the image sector of the tile's row 0 and (for confirmation) that row's bytes
  uint64_t my_sector = 0;
  const uint8_t* my_bytes = nullptr;
  if (my_n) {
    const uint64_t my_u = u0 + lane, ctile = my_u / kW;
    const Segment* const segs = p.segs.get();
    const Segment& sg = segs[find_segment(segs, p.segs.n, ctile)];
    const uint64_t row_first = (ctile - sg.tile_base) * T + (my_u % kW) * 32;  // within the segment
    my_sector = sg.sector_base + row_first;
    if (p.confirm) my_bytes = sg.bytes + row_first * kSector;
  }
  uint32_t carry = 0, carry_b = 32;  // triples of tile carry_b's records in earlier passes
  for (uint32_t q0 = 0; q0 < n_rec; q0 += 32) {
    const uint32_t q = q0 + lane;
    const bool act = q < n_rec;
    // the record's tile: the last lane b whose first record is at or before q
    uint32_t b = 0;
#pragma unroll
    for (uint32_t step = 16; step > 0; step >>= 1)
      if (__shfl_sync(kFull, my_first, b + step) <= q) b += step;
    const uint32_t i = q - __shfl_sync(kFull, my_first, b);
    const uint64_t off_b = __shfl_sync(kFull, my_off, b);
    const uint64_t sector_b = __shfl_sync(kFull, my_sector, b);
    const uint8_t* bytes_b =
        reinterpret_cast<const uint8_t*>(__shfl_sync(kFull, reinterpret_cast<uintptr_t>(my_bytes), b));
    uint4 rec = make_uint4(0, 0, 0, 0);
    if (act) rec = p.hit_rec[(u0 + b) * 32 + i];
    // triples of the records before this one in its tile: a scan over the lanes of the same tile
    uint32_t sum = rec.w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(kFull, sum, d);
      const uint32_t vb = __shfl_up_sync(kFull, b, d);
      if (lane >= (uint32_t)d && vb == b) sum += v;
    }
    const uint32_t before = sum - rec.w + (b == carry_b ? carry : 0u);
    const uint32_t last_b = __shfl_sync(kFull, b, 31);
    const uint32_t last_sum = __shfl_sync(kFull, sum, 31);
    carry = last_sum + (last_b == carry_b ? carry : 0u);
    carry_b = last_b;
    if (!act) continue;
    uint64_t o = off_b + before;
    const bool check = rec.w < rec.z;
    const uint8_t* mine = check ? bytes_b + (uint64_t)rec.x * kSector : nullptr;
    for (uint32_t k = 0; k < rec.z; k++) {
      if (check && !sectors_equal(mine, p.confirm + (uint64_t)(rec.y + k) * kSector)) continue;
      if (o < p.out_cap) {
        const uint2 pf = p.postings[rec.y + k];
        p.out[o] = MatchOut{sector_b + rec.x, pf.x, pf.y};
      } else {
        atomicOr(p.status, kStOverflow);
      }
      o++;
    }
  }
}

// The hits of the group's tiles and their numbering: returns their number; my_n, my_first: this
// lane's tile.
__device__ __forceinline__ uint32_t group_hits(const CompactParams& p, uint64_t u0, uint32_t& my_n,
                                               uint32_t& my_first) {
  const uint32_t lane = threadIdx.x & 31;
  my_n = u0 + lane < p.n_out_tiles ? p.tile_nhit[u0 + lane] : 0u;
  uint32_t incl = my_n;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= (uint32_t)d) incl += v;
  }
  my_first = incl - my_n;
  return __shfl_sync(0xFFFFFFFFu, incl, 31);
}

// The second pass over offsets made before (larger scans). When the scan before it on the stream
// failed (a wait timed out or a lookup ran past the probe bound: its hit records are not to be
// trusted), the pass writes nothing.
template <int T>
__global__ void expand_kernel(const __grid_constant__ CompactParams p) {
  if (*(volatile const uint32_t*)p.status & (kStTimeout | kStProbeBound | kStBadTable)) return;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  for (uint64_t u0 = ((uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; u0 < p.n_out_tiles;
       u0 += warps * 32) {
    uint32_t my_n, my_first;
    const uint32_t n_rec = group_hits(p, u0, my_n, my_first);
    if (n_rec == 0u) continue;
    expand_group<T>(p, u0, my_n, my_first, n_rec, my_n ? p.tile_off[u0 + (threadIdx.x & 31)] : 0ull);
  }
}

// Offsets and expansion in one launch, for scans of at most kFinishTiles output tiles: every block
// sums all groups of 32 tiles and scans the sums itself (at most 1 MB, from L2), then expands its
// share of the groups; block 0 writes the total and the segments' offsets. One launch in place of a
// memset and three, whose gaps and latencies are what a small scan's second half consists of: 64 KiB
// 6.6 us against 11.9 and the gaps (call 79 against 89 us), 1 GiB (65,540 tiles) 17.7 against 18.2
// and the gaps (call 322 against 331). A warp loads eight groups' counts at a time: one by one the
// 1 GiB scan's took 38 us. Above kFinishTiles every block's pass over all tiles costs more than
// the three launches.
constexpr uint64_t kFinishTiles = 1ull << 17;
constexpr int kFinishThreads = 1024;

template <int T>
__global__ void __launch_bounds__(kFinishThreads) finish_kernel(const __grid_constant__ CompactParams p) {
  extern __shared__ uint64_t s_group[];  // per group: its triples, then the triples before it
  __shared__ uint64_t s_warp[33];
  constexpr uint32_t kFull = 0xFFFFFFFFu;
  constexpr uint32_t kWarps = kFinishThreads / 32;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_groups = (uint32_t)((p.n_out_tiles + 31) / 32);
  constexpr uint32_t kAhead = 8;  // groups whose counts a warp loads at a time
  for (uint32_t g0 = warp; g0 < n_groups; g0 += kWarps * kAhead) {
    uint64_t n[kAhead];
#pragma unroll
    for (uint32_t k = 0; k < kAhead; k++) {
      const uint64_t u = 32ull * (g0 + k * kWarps) + lane;
      n[k] = u < p.n_out_tiles ? p.tile_ntrip[u] : 0ull;
    }
#pragma unroll
    for (uint32_t k = 0; k < kAhead; k++) {
      uint64_t sum = __reduce_add_sync(kFull, (uint32_t)n[k] & 0xFFFFFFu);
      if (__any_sync(kFull, (n[k] >> 24) != 0u)) {  // keys with very many postings
        uint64_t high = n[k] >> 24;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) high += __shfl_xor_sync(kFull, (unsigned long long)high, d);
        sum += high << 24;
      }
      if (lane == 0 && g0 + k * kWarps < n_groups) s_group[g0 + k * kWarps] = sum;
    }
  }
  __syncthreads();
  // exclusive scan of the groups' sums: `per` consecutive ones a thread
  const uint32_t per = (n_groups + kFinishThreads - 1) / kFinishThreads;
  uint64_t mine = 0;
  for (uint32_t k = 0; k < per; k++)
    if (tid * per + k < n_groups) mine += s_group[tid * per + k];
  uint64_t incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t v = __shfl_up_sync(kFull, (unsigned long long)incl, d);
    if (lane >= (uint32_t)d) incl += v;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const uint64_t w = s_warp[lane];
    uint64_t wi = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint64_t v = __shfl_up_sync(kFull, (unsigned long long)wi, d);
      if (lane >= (uint32_t)d) wi += v;
    }
    s_warp[lane] = wi - w;
    if (lane == 31) s_warp[32] = wi;
  }
  __syncthreads();
  uint64_t run = s_warp[warp] + incl - mine;
  for (uint32_t k = 0; k < per; k++) {
    if (tid * per + k >= n_groups) break;
    const uint64_t v = s_group[tid * per + k];
    s_group[tid * per + k] = run;
    run += v;
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    if (tid == 0) *p.total = s_warp[32];
    const Segment* const segs = p.segs.get();
    for (uint32_t s = tid; s < p.segs.n; s += kFinishThreads) {
      const uint64_t u = segs[s].tile_base * (T / 32);
      uint64_t off = u < p.n_out_tiles ? s_group[u / 32] : s_warp[32];
      if (u < p.n_out_tiles)
        for (uint64_t q = u & ~31ull; q < u; q++) off += p.tile_ntrip[q];
      p.seg_off[s] = off;
    }
  }
  const bool failed = *(volatile const uint32_t*)p.status & (kStTimeout | kStProbeBound | kStBadTable);
  uint32_t hits = 0;
  for (uint32_t g = blockIdx.x * kWarps + warp; g < n_groups && !failed; g += gridDim.x * kWarps) {
    const uint64_t u0 = 32ull * g;
    uint32_t my_n, my_first;
    const uint32_t n_rec = group_hits(p, u0, my_n, my_first);
    if (n_rec == 0u) continue;
    hits += n_rec;
    uint64_t off = my_n ? p.tile_ntrip[u0 + lane] : 0ull;  // a tile without hits has no triples
    const uint64_t own = off;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint64_t v = __shfl_up_sync(kFull, (unsigned long long)off, d);
      if (lane >= (uint32_t)d) off += v;
    }
    expand_group<T>(p, u0, my_n, my_first, n_rec, s_group[g] + off - own);
  }
  if (p.nhit_sum && lane == 0 && hits) atomicAdd(p.nhit_sum, (unsigned long long)hits);
}

}  // namespace cvk
