// Second half of the match compaction: the per-tile triple counts of the scan are turned into
// output offsets by an exclusive scan, and every hit record of every tile is expanded into
// its (disk_sector, file_id, file_sector) triples. Tiles are in sector order, the records of a
// tile are in sector order (ballot ranks), and each digest's postings are sorted by
// (file_id, file_sector), so the output is sorted without a sort. (The paper's Section 3.2 writes
// matches to a host-visible buffer in no stated order; the sorted triple list is this library's
// output format.)
#pragma once
#include <stdint.h>

#include "cv_internal.h"

namespace cvk {

// Exclusive scan of per-tile counts in one pass, for the serving loop and the fragment scans: each
// block scans a chunk, adds its predecessors' published sums (decoupled look-back, every wait
// bounded) and writes the offsets of the segments that begin in the chunk. (This kernel is in
// kernels_scan.cu; this header holds the passes instantiated with each configuration.)
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
  uint32_t all_or_none;        // finish_kernel: nothing is written, nor tried, when out_cap is too little for all
  uint32_t* status;
  const uint64_t* tile_off;    // expand_kernel: output offset per tile
  const unsigned long long* group_sum;  // finish_kernel: triples per 2^group_log2 tiles
  uint32_t group_log2;
  uint32_t n_groups;           // at most kFinishGroups
  uint64_t* seg_off;           // out, the offset of every segment's first tile
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
// A record's postings are written by one lane, bound by the latency of a posting's load while the next
// had to wait for the store before it; loaded as read-only data, four in flight, 32 MiB with 128 copies
// of each sector take 207 us instead of 573.
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
    const uint2* const post = p.postings + rec.y;
    MatchOut* const out = p.out + o;
    const uint64_t room = o < p.out_cap ? p.out_cap - o : 0ull;
    if (rec.w > room) atomicOr(p.status, kStOverflow);
    if (rec.w == rec.z) {
      const uint32_t n = rec.w < room ? rec.w : (uint32_t)room;
#pragma unroll 4
      for (uint32_t k = 0; k < n; k++) {
        const uint2 pf = __ldg(post + k);
        out[k] = MatchOut{sector_b + rec.x, pf.x, pf.y};
      }
    } else {
      const uint8_t* mine = bytes_b + (uint64_t)rec.x * kSector;
      uint32_t n = 0;
      for (uint32_t k = 0; k < rec.z; k++) {
        if (!sectors_equal(mine, p.confirm + (uint64_t)(rec.y + k) * kSector)) continue;
        if (n < room) {
          const uint2 pf = __ldg(post + k);
          out[n] = MatchOut{sector_b + rec.x, pf.x, pf.y};
        }
        n++;
      }
    }
  }
}

// The numbering of the hits of the warp's tiles (this lane's has my_n): returns their number;
// my_first: the first of this lane's.
__device__ __forceinline__ uint32_t group_hits(uint32_t my_n, uint32_t& my_first) {
  const uint32_t lane = threadIdx.x & 31;
  uint32_t incl = my_n;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= (uint32_t)d) incl += v;
  }
  my_first = incl - my_n;
  return __shfl_sync(0xFFFFFFFFu, incl, 31);
}

// The expansion alone, over offsets made before (the serving loop, whose host reads the counts in
// between). When the scan before it on the stream failed (a wait timed out or a lookup ran past the
// probe bound: its hit records are not to be trusted), the pass writes nothing.
template <int T>
__global__ void expand_kernel(const __grid_constant__ CompactParams p) {
  if (*(volatile const uint32_t*)p.status & (kStTimeout | kStProbeBound | kStBadTable)) return;
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  for (uint64_t u0 = ((uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; u0 < p.n_out_tiles;
       u0 += warps * 32) {
    const uint64_t u = u0 + (threadIdx.x & 31);
    const uint32_t my_n = u < p.n_out_tiles ? p.tile_nhit[u] : 0u;
    uint32_t my_first;
    const uint32_t n_rec = group_hits(my_n, my_first);
    if (n_rec == 0u) continue;
    expand_group<T>(p, u0, my_n, my_first, n_rec, my_n ? p.tile_off[u] : 0ull);
  }
}

// Offsets and expansion in one launch. The scan has summed its triples by groups of tiles (an atomic
// for a tile that has any); every block scans these sums, at most kFinishGroups, and takes groups: a
// thread per tile, 512 at a time, their counts scanned over the block, then a warp per 32 tiles
// expands. What bounds it is latency: the sums, the counts, then for tiles with hits the record, the
// posting and the write, each waiting for the one before it; so the counts of the next 512 tiles are
// loaded before these are expanded (without that 7.2, 10.9 and 74 us where the last column says 6.2,
// 9.6 and 64), and a group without triples is passed over. It took the place of a memset and three
// launches (look-back offset scan, segments' offsets, expansion), the gaps between them not counted
// here:            three launches       this one
//   64 KiB         4.2 + 2.8 + 4.9 us   6.2 us
//   1 GiB          8.2 + 2.7 + 7.3      9.1
//   2 GiB, CRC64   10.5 + 2.6 + 7.7     9.6
//   32 GiB, 1,000,000 matches: 64
// A group is what one block expands, so few of them leave SMs idle where most sectors of a small image
// match: a group has 32 tiles, or as many more (up to 512) as leave two groups per SM; 512 from 2.3 GiB to
// 32 GiB, more above, so that the sums' scan stays at most 4,096 words a block. Offsets and expansion, us,
// with groups of 512 tiles at least, and so (copies: of each matching sector in the master files):
//   8 MiB, all of it matches, 16 copies    323    97
//   32 MiB, 128 copies                     2,379  573
//   256 MiB, 8 copies                      179    72
//   1 GiB, one sector in 64 matches        19     19 to 21
// (608 groups: 122 at 256 MiB, 23 at 1 GiB.) A block whose group has fewer tiles than threads has idle
// warps, which costs nothing there.
constexpr uint32_t kFinishGroups = 4096;
constexpr int kFinishThreads = 512;
constexpr uint32_t kFinishMinLog2 = 5;    // a warp's tiles
constexpr uint32_t kFinishChunkLog2 = 9;  // groups of as many tiles or more are whole chunks of kFinishThreads
constexpr uint32_t kFinishFew = 304;      // groups of fewer tiles than a chunk, at most
static_assert((1 << kFinishChunkLog2) == kFinishThreads, "chunks of a tile per thread");

// The group size for n output tiles.
inline uint32_t finish_group_log2(uint64_t n) {
  uint32_t l = kFinishMinLog2;
  while (((n + (1ull << l) - 1) >> l) > (l < kFinishChunkLog2 ? kFinishFew : kFinishGroups)) l++;
  return l;
}
inline uint32_t finish_groups(uint64_t n) {
  const uint32_t l = finish_group_log2(n);
  return (uint32_t)((n + (1ull << l) - 1) >> l);
}

// Exclusive scan of x over the kFinishThreads threads of a block; *total gets the sum. buf: 17 words.
__device__ __forceinline__ uint64_t finish_scan(uint64_t x, uint64_t* buf, uint64_t* total) {
  constexpr uint32_t kFull = 0xFFFFFFFFu;
  constexpr int kWarps = kFinishThreads / 32;
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t incl = x;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t v = __shfl_up_sync(kFull, (unsigned long long)incl, d);
    if (lane >= (uint32_t)d) incl += v;
  }
  if (lane == 31) buf[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const uint64_t w = lane < (uint32_t)kWarps ? buf[lane] : 0ull;
    uint64_t wi = w;
#pragma unroll
    for (int d = 1; d < kWarps; d <<= 1) {
      const uint64_t v = __shfl_up_sync(kFull, (unsigned long long)wi, d);
      if (lane >= (uint32_t)d) wi += v;
    }
    if (lane < (uint32_t)kWarps) buf[lane] = wi - w;
    if (lane == kWarps - 1) buf[kWarps] = wi;
  }
  __syncthreads();
  *total = buf[kWarps];
  const uint64_t r = buf[warp] + incl - x;
  __syncthreads();  // buf may be used again
  return r;
}

template <int T>
__global__ void __launch_bounds__(kFinishThreads) finish_kernel(const __grid_constant__ CompactParams p) {
  __shared__ uint64_t s_group[kFinishGroups];  // triples before the group
  __shared__ uint64_t s_off[kFinishThreads];   // offsets of the chunk's tiles
  __shared__ uint64_t s_buf[kFinishThreads / 32 + 1];
  constexpr uint32_t kPer = kFinishGroups / kFinishThreads;
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  uint64_t g[kPer], mine = 0, total;
#pragma unroll
  for (uint32_t k = 0; k < kPer; k++) {
    g[k] = tid * kPer + k < p.n_groups ? p.group_sum[tid * kPer + k] : 0ull;
    mine += g[k];
  }
  uint64_t run = finish_scan(mine, s_buf, &total);
#pragma unroll
  for (uint32_t k = 0; k < kPer; k++) {
    s_group[tid * kPer + k] = run;
    run += g[k];
  }
  const bool no_room = p.all_or_none && total > p.out_cap;
  if (blockIdx.x == 0 && tid == 0) {
    *p.total = total;
    if (no_room) atomicOr(p.status, kStOverflow);
  }
  const Segment* const segs = p.segs.get();
  const bool failed = *(volatile const uint32_t*)p.status & (kStTimeout | kStProbeBound | kStBadTable);
  uint32_t hits = 0;
  __syncthreads();
  // The block's chunks one after another; a chunk's counts are loaded while the one before it is
  // expanded.
  uint32_t gi = blockIdx.x;
  uint64_t c0 = (uint64_t)gi << p.group_log2;
  uint64_t next_trip = 0, next_at = 0;
  uint32_t next_hit = 0;
  const auto load = [&](uint32_t g_, uint64_t c_) {
    const uint64_t u = c_ + tid;
    const bool in = g_ < p.n_groups && u < min(((uint64_t)g_ + 1) << p.group_log2, p.n_out_tiles);
    next_trip = in ? p.tile_ntrip[u] : 0ull;
    next_hit = in ? p.tile_nhit[u] : 0u;
  };
  if (gi < p.n_groups) next_at = s_group[gi];
  load(gi, c0);
  while (gi < p.n_groups) {
    const uint64_t at = next_at, trip = next_trip, first_tile = c0;
    const uint32_t my_n = next_hit;
    const uint64_t end = min(((uint64_t)gi + 1) << p.group_log2, p.n_out_tiles);
    const bool empty = (gi + 1 < p.n_groups ? s_group[gi + 1] : total) == s_group[gi];
    c0 += kFinishThreads;
    const bool same_group = c0 < end;
    if (!same_group) {
      gi += gridDim.x;
      c0 = (uint64_t)gi << p.group_log2;
    }
    load(gi, c0);
    uint64_t sum = 0, off = at;
    if (!empty) off += finish_scan(trip, s_buf, &sum);
    next_at = same_group ? at + sum : gi < p.n_groups ? s_group[gi] : 0ull;
    if (p.segs.n > 1 || first_tile == 0) {  // segments that begin in this chunk
      s_off[tid] = off;
      __syncthreads();
      const uint64_t c1 = min(first_tile + kFinishThreads, end);
      uint32_t lo = 0, hi = p.segs.n;  // the first segment at or after the chunk's first tile
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (segs[mid].tile_base * (T / 32) < first_tile) lo = mid + 1; else hi = mid;
      }
      for (uint32_t s = lo + tid; s < p.segs.n; s += kFinishThreads) {
        const uint64_t first = segs[s].tile_base * (T / 32);
        if (first >= c1) break;
        p.seg_off[s] = s_off[first - first_tile];
      }
      __syncthreads();
    }
    if (!empty && !failed) {
      uint32_t my_first;
      const uint32_t n_rec = group_hits(my_n, my_first);
      if (n_rec && !no_room) expand_group<T>(p, first_tile + tid - lane, my_n, my_first, n_rec, off);
      hits += n_rec;
    }
  }
  if (p.nhit_sum && lane == 0 && hits) atomicAdd(p.nhit_sum, (unsigned long long)hits);
}

}  // namespace cvk
