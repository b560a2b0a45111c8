// Kernel configurations of the scan, exported by kernels_scan.cu to the host runtime.
#pragma once
#include <stdint.h>

#include "cv_internal.h"

namespace cvk {

struct ScanCfg {
  const char* name;
  int T;        // sectors per tile; T / 32 output tiles per tile
  int SPT;      // sectors per hashing thread
  int threads;  // block size: T / SPT hashing threads + one producer warp
  int NS;       // shared-memory ring stages
  int BOXB;   // bytes of each sector row per stage (64 or 128)
  const void* scan_fn[8];    // scan_kernel per table kind (table_kind); null: not built for it
  const void* digest_fn[4];  // digest mode, per signature (kSig*)
  const void* expand_fn;     // expand_kernel<T>
  const void* finish_fn;     // finish_kernel<T>
  uint32_t smem;             // dynamic shared memory bytes
};

const ScanCfg* scan_configs(int* n);
// The configurations of each instantiation unit, in table order (scan_cfgs_{a,b,c}.cu).
const ScanCfg* scan_cfgs_a(int* n);
const ScanCfg* scan_cfgs_b(int* n);
const ScanCfg* scan_cfgs_c(int* n);

// Scan kernels are selected by signature and by how the table is looked up: kind = sig for a walk over
// the slots, sig + 4 for the others (bisection, walk over the tags). The tags' walk in the kernels of
// the slots' walk made every scan with a filter 4% slower (0.408 to 0.424 ms for 2 GiB; as a function
// that is called 0.9%), by the registers and code it adds.
constexpr int kTableKinds = 8;
inline int table_kind(const TableView& t) { return (int)t.sig + (t.layout == kLayoutSorted || t.tags ? 4 : 0); }

// Configuration cfg_i if it has a scan kernel for table kind `kind` (table_kind), else the
// default one (index 0, which has every kind); *used receives the index in use.
const ScanCfg& scan_config_for(int cfg_i, int kind, int* used);
// The default scan configuration for a table kind and a number of sectors (the fastest measured).
int preferred_config(int kind, uint64_t sectors, int sms);
// Configuration cfg_i (-1: the preferred one for the signature and the sectors) if it has a
// digest-mode kernel for signature sig, else the first one.
const ScanCfg& digest_config_for(int cfg_i, int sig, uint64_t sectors, int sms, int* used);

// The expand pass (see expand_kernel). Returns a CUDA error code.
struct CompactParams;
int launch_expand(const ScanCfg& cfg, const CompactParams& p, int sms, void* stream);
// Offsets and expansion in one launch (see finish_kernel).
int launch_finish(const ScanCfg& cfg, const CompactParams& p, int sms, void* stream);
// The tables' side of CompactParams.
void compact_table(CompactParams* p, const TableView& tab);

// Scratch (u64 words) the offset pass (serving loop, fragment scans) needs for n tiles.
uint64_t tile_offsets_scratch_words(uint64_t n_tiles);

// tile_off[i] = sum of tile_ntrip[0..i) over the n_tiles output tiles; *total = sum of all;
// seg_off[s] = offset of segment s's first output tile (segment tile_base * scale). scratch:
// tile_offsets_scratch_words(n_tiles) u64 words. status: the scan's status word (kStTimeout if
// a wait of the pass gives up). zeroed: the scratch is zero already. Returns a CUDA error code.
int launch_tile_offsets(const uint64_t* tile_ntrip, uint64_t n_tiles, uint64_t* tile_off, const SegList& segs,
                        uint32_t scale, uint64_t* seg_off, uint64_t* total, uint64_t* scratch, void* stream,
                        uint32_t* status, bool zeroed = false);

// ---------------------------------------------------------------- fragment scans (Section 5)
uint64_t frag_windows(uint64_t n_bytes);       // 64-byte windows at 4-byte offsets in n_bytes
uint64_t frag_tiles(int sig, uint64_t n_bytes);  // tiles of sig's fragment kernels over those windows
// Which filters and count kernel a table with n_keys keys has.
enum : int { kFragFewKeys = 0, kFragManyKeys = 1, kFragMostKeys = 2, kFragKeyClasses = 3 };
int frag_key_class(int sig, uint64_t n_keys);
bool frag_sig_supported(int sig);         // MD5, MD5 without padding, djb2-64

// Key words and exclusion flags of n master fragments at arena (64 bytes each, 16-byte aligned).
int frag_digests(int sig, const uint8_t* arena, uint64_t n, uint4* dig, uint8_t* trivial, int sms, void* stream);
// The filters of a fragment table (zeroed by the caller): the one-word Bloom filter (words, null
// for none; mask = words - 1) and the shared-memory filter l1 (kFragL1Bytes).
int frag_bloom(int sig, const uint4* slots, uint32_t n_slots, uint64_t n_keys, uint32_t* words, uint32_t mask,
               uint32_t* l1, int sms, void* stream);
// The images of a scan that have a tile, in order: their tiles are numbered through, an image's begin at
// tile_base. Up to kInlineSegs of them travel in the kernels' parameters, as SegList's segments do.
struct FragImage {
  const uint8_t* data;  // device memory, 16-byte aligned
  uint64_t n_bytes, n_windows, tile_base;
};
struct FragImages {
  const FragImage* dev;  // device memory; not used (may be null) when n <= kInlineSegs
  uint32_t n;
  uint32_t pad;
  FragImage in[kInlineSegs];
  __host__ __device__ const FragImage* get() const { return n <= kInlineSegs ? in : dev; }
};
FragImages frag_images(const FragImage* host, const FragImage* dev, size_t n);

// The hit list of a scan: tiles has room for every tile, masks (32 words per tile) for the first
// mask_tiles that are listed.
struct FragHits {
  uint32_t* tiles;
  uint32_t* masks;
  uint64_t mask_tiles;
  uint32_t* count;
};
constexpr uint64_t kFragMaskTiles = 1ull << 22;
// Triples per tile of the images (n_tiles in all) into tile_ntrip and their hit list (*hits.count zero
// before); djb2 candidates dropped by the byte comparison are added to *rejected (when non-null).
int frag_count(const TableView& tab, const FragImages& images, uint64_t n_tiles, uint64_t* tile_ntrip, const FragHits& hits,
               uint32_t* status, unsigned long long* rejected, int sms, void* stream);
// The 16-byte key of every 64-byte window at a 4-byte offset of a device image, through the
// fragment kernels' own signature code (MD5, MD5 without padding, rolled djb2-64).
int frag_window_sigs(int sig, const uint8_t* image, uint64_t n_bytes, uint4* out, int sms, void* stream);
// The triples of the listed tiles, at out[tile_off[tile]..]; none when *total (device memory, the triples
// of all images) is above out_cap.
int frag_emit(const TableView& tab, const FragImages& images, uint64_t n_tiles, const uint64_t* tile_off,
              const uint64_t* total, const FragHits& hits, MatchOut* out, uint64_t out_cap, uint32_t* status, int sms,
              void* stream);

// The offset scan's look-back wait running out (words: lookback_selftest_words() u64).
int launch_lookback_selftest(uint64_t* words, uint32_t* status, uint64_t timeout_ns, void* stream);
constexpr uint64_t lookback_selftest_words() { return 4 * 4096 + 4; }

// One block whose single waiting thread waits on an mbarrier nothing completes (bounded by
// timeout_ns): the status word gets the timeout bit. Returns a CUDA error code.
int launch_wait_selftest(uint32_t* status, uint64_t timeout_ns, void* stream);

}  // namespace cvk
