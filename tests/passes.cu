// The library's device passes driven one by one with scratch that a caller of the C ABI has no say over:
// the room of the output, and how many hit-list entries of a fragment scan have masks. Built and used by
// test_gpu_passes.py against libcv.so.
#include <cuda_runtime.h>
#include <string.h>

#include <vector>

#include "compact.cuh"
#include "runtime.h"

using namespace cvk;

namespace {

struct Bufs {
  std::vector<void*> owned;
  ~Bufs() {
    cudaDeviceSynchronize();
    for (void* p : owned) cudaFree(p);
  }
  template <class T>
  int get(T** out, uint64_t n) {
    void* p = nullptr;
    CV_CUDA(cudaMalloc(&p, n * sizeof(T) + 16));
    owned.push_back(p);
    CV_CUDA(cudaMemset(p, 0, n * sizeof(T) + 16));
    *out = static_cast<T*>(p);
    return CV_OK;
  }
};

}  // namespace

extern "C" {

// A scan of n sectors at image (device) with the finishing pass's room for cap triples at out.
// h: total, status, sectors with a match.
int passes_scan(const cv_master* m, const void* image, uint64_t n, uint64_t cap, int all_or_none, void* out, uint64_t* h) {
  DevCtx* ctx;
  TableView tab;
  int dev, cfg_i;
  CV_TRY(get_ctx(&ctx));
  CV_TRY(master_view(m, &tab, &dev));
  const ScanCfg& cfg = scan_config_for(ctx->default_config(table_kind(tab), n), table_kind(tab), &cfg_i);
  Job job;
  CV_TRY(job.add(ctx, cfg, image, n, 0, 0, false));
  if (job.segs.size() > kInlineSegs) return CV_EINVAL;
  const uint64_t tiles = job.n_tiles * (uint64_t)(cfg.T / 32);
  Bufs b;
  ScanParams p;
  memset(&p, 0, sizeof p);
  p.tab = tab;
  CV_TRY(b.get(&p.hit_rec, tiles * 32));
  CV_TRY(b.get(&p.tile_nhit, tiles));
  CV_TRY(b.get(&p.tile_ntrip, tiles));
  CV_TRY(b.get(&p.group_sum, finish_groups(tiles)));
  p.group_log2 = finish_group_log2(tiles);
  uint64_t* words;  // segment offsets, total, status, sectors with a match
  CV_TRY(b.get(&words, job.segs.size() + 3));
  uint64_t* const total = words + job.segs.size();
  p.status = (uint32_t*)(total + 1);
  CV_CUDA(cudaDeviceSynchronize());
  CV_TRY(launch_range(ctx, cfg_i, false, job, nullptr, 0, job.segs.size(), p, nullptr));
  CompactParams cp;
  memset(&cp, 0, sizeof cp);
  compact_table(&cp, tab);
  cp.hit_rec = p.hit_rec;
  cp.tile_nhit = p.tile_nhit;
  cp.tile_ntrip = p.tile_ntrip;
  cp.n_out_tiles = tiles;
  cp.segs = seg_list(job.segs.data(), nullptr, job.segs.size());
  cp.out = (MatchOut*)out;
  cp.out_cap = cap;
  cp.all_or_none = (uint32_t)all_or_none;
  cp.status = p.status;
  cp.group_sum = p.group_sum;
  cp.group_log2 = p.group_log2;
  cp.n_groups = finish_groups(tiles);
  cp.seg_off = words;
  cp.total = total;
  cp.nhit_sum = (unsigned long long*)(total + 2);
  CV_CUDA((cudaError_t)launch_finish(cfg, cp, ctx->sms, nullptr));
  CV_CUDA(cudaMemcpy(h, total, 24, cudaMemcpyDeviceToHost));
  return CV_OK;
}

// A fragment scan of n images (device): masks for mask_tiles listed tiles, room for cap triples at out.
// h: total, status, then the images' first triples.
int passes_fragments(const cv_master* m, const void* const* images, const uint64_t* bytes, uint32_t n, uint64_t mask_tiles,
                     uint64_t cap, void* out, uint64_t* h) {
  DevCtx* ctx;
  TableView tab;
  int dev;
  CV_TRY(get_ctx(&ctx));
  CV_TRY(master_view(m, &tab, &dev));
  std::vector<uint64_t> base(n + 1, 0);
  std::vector<Segment> segs(n);
  for (uint32_t i = 0; i < n; i++) {
    base[i + 1] = base[i] + frag_tiles((int)tab.sig, bytes[i]);
    memset(&segs[i], 0, sizeof(Segment));
    segs[i].tile_base = base[i];
  }
  if (n > kInlineSegs) return CV_EINVAL;
  const uint64_t tiles = base[n];
  Bufs b;
  uint64_t *ntrip, *off, *words, *scratch;  // words: total, status, segment offsets, listed tiles
  FragHits hits;
  CV_TRY(b.get(&ntrip, tiles));
  CV_TRY(b.get(&off, tiles));
  CV_TRY(b.get(&words, 3 + n));
  CV_TRY(b.get(&scratch, tile_offsets_scratch_words(tiles)));
  CV_TRY(b.get(&hits.tiles, tiles));
  hits.mask_tiles = mask_tiles < tiles ? mask_tiles : tiles;
  CV_TRY(b.get(&hits.masks, hits.mask_tiles * 32));
  uint32_t* const status = (uint32_t*)(words + 1);
  hits.count = (uint32_t*)(words + 2 + n);
  std::vector<FragImage> list;
  for (uint32_t i = 0; i < n; i++) list.push_back(FragImage{(const uint8_t*)images[i], bytes[i], frag_windows(bytes[i]), base[i]});
  const FragImages scanned = frag_images(list.data(), nullptr, n);
  CV_CUDA(cudaDeviceSynchronize());
  CV_CUDA((cudaError_t)frag_count(tab, scanned, tiles, ntrip, hits, status, nullptr, ctx->sms, nullptr));
  CV_CUDA((cudaError_t)launch_tile_offsets(ntrip, tiles, off, seg_list(segs.data(), nullptr, n), 1, words + 2, words,
                                           scratch, nullptr, status));
  CV_CUDA((cudaError_t)frag_emit(tab, scanned, tiles, off, words, hits, (MatchOut*)out, cap, status, ctx->sms, nullptr));
  CV_CUDA(cudaMemcpy(h, words, (2 + n) * 8, cudaMemcpyDeviceToHost));
  return CV_OK;
}

}  // extern "C"
