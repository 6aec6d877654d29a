// Allocation-free forward render.
//
// Some callers cannot allocate device memory: a plugin or engine integration that runs
// inside a host application which owns the whole device heap and only hands it buffers,
// or code under a memory budget enforced by an outer allocator, where a cudaMalloc from a
// library is forbidden.  For them raygs_render_noalloc renders a small scene with every
// intermediate buffer (per-view records, sort keys, instance lists, tile ranges, counters)
// carved from one file-scope device array of fixed size: the library allocates nothing,
// neither device memory (no cudaMalloc/cudaFree) nor host heap.
//
// The array is a module-scope __device__ variable: every GPU that loads this library keeps
// kNoAllocScratchBytes of device memory reserved for it until the process exits.
#include <algorithm>

#include "raygs_internal.cuh"

namespace raygs {

constexpr size_t kNoAllocScratchBytes = RAYGS_NOALLOC_SCRATCH_BYTES;
__device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

}  // namespace raygs

using namespace raygs;

namespace {

// Device address of the scratch array in the current device's context.  Host code cannot
// use the symbol itself (it names a host-side shadow).  The lookup is made on every call:
// it is cheap once the module is loaded, and it stays right if the context was destroyed
// and created again (cudaDeviceReset), where the array may sit at a new address.  The
// first call on a device loads the module there.
raygs_status scratch_for_current_device(void **out) {
  void *p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
  if (e != cudaSuccess || !p) {
    note_cuda_error(e);
    return RAYGS_ERR_CUDA;
  }
  *out = p;
  return RAYGS_OK;
}

// Size check: the fixed part must fit; the rest of the array bounds the tile rows and instances.  What only
// makes a pass faster (the row pass's head chunks, the tiles by class on small batches, short chunks of
// wide views in the list pass) is left out of a batch that would otherwise not fit, or keep less than two
// thirds of the capacity.
bool fit_scratch(Work &w) {
  const uint32_t rows_short = list_rows_short(w.max_tiles_x);
  const struct { int heads; bool order; uint32_t list_lo; } keep[] = {
      {kHeadChunks, w.tiles <= 8192, kListRowsLo}, {16, false, rows_short}, {0, false, rows_short}};
  LayoutOptions opt;
  opt.tile_stop = false;
  opt.bin_once = true;
  opt.short_chunks = w.short_chunks = false;
  auto layout = [&](int64_t cap) {
    w.cap = cap;
    w.L = make_layout(w.n_views, w.n, w.tiles, w.trows, cap, w.num_sms, w.max_tiles_x, w.max_rows, opt);
    return w.L.total <= kNoAllocScratchBytes;
  };
  double room = 0.0;
  // The capacity that the i-th choice leaves, but for the rounding of the buffers.
  auto guess = [&](int i) {
    opt.tile_order = keep[i].order;
    opt.heads = w.heads = keep[i].heads;
    opt.list_lo = w.list_lo = keep[i].list_lo;
    layout(0);
    room = double(kNoAllocScratchBytes) - double(w.L.total);
    // the column counts: up to so many bytes per unit of capacity, and no more than so many in all
    const double per_unit = 4.0 * w.max_tiles_x / w.list_lo, in_all = 4.0 * w.max_tiles_x * list_target(w.num_sms);
    return int64_t(std::max(room / (kBytesPerCapacity + per_unit), (room - in_all) / kBytesPerCapacity));
  };
  auto fits = [&](int64_t cap) {
    while (cap > 0 && !layout(cap)) cap -= 256;
    return cap > 0;
  };
  // the usual case: two thirds of all that is left besides what the choices differ in
  int64_t cap = guess(0);
  const double extras = 4.0 * kTileClasses * double(w.tiles) + double(w.L.rows - w.L.cnt1);
  if (cap > 0 && 3.0 * kBytesPerCapacity * double(cap) >= 2.0 * (room + extras) && fits(cap)) return true;
  const int64_t most = guess(2);
  for (int i = 0; i < 3 && most > 0; ++i)
    if (3 * (cap = guess(i)) >= 2 * most && fits(cap)) return true;
  return false;
}

}  // namespace

extern "C" raygs_status raygs_render_noalloc(const raygs_camera *cams, int32_t n_views, const raygs_scene *scene,
                                             const raygs_config *cfg_in, float *rgb, float *T_final,
                                             int32_t *n_contrib, void *stream) {
  if (!cams || !scene || !rgb || n_views < 1 || n_views > RAYGS_MAX_VIEWS) return RAYGS_ERR_INVALID_ARG;
  raygs_config cfg;
  if (cfg_in) cfg = *cfg_in; else raygs_config_default(&cfg);
  cfg.enable_backward = 0;
  if (!config_valid(cfg)) return RAYGS_ERR_INVALID_ARG;
  const int64_t n = scene->n;
  if (n < 0 || n >= (int64_t(1) << 31)) return RAYGS_ERR_INVALID_ARG;
  raygs_status s = scene_valid(scene, n);
  if (s != RAYGS_OK) return s;

  // Per-view constants, on the stack (no heap).
  DevCam dc[RAYGS_MAX_VIEWS];
  int64_t tiles = 0, trows = 0, pixels = 0;
  int max_tx = 0, max_rows = 0;
  if (!plan_views(cams, n_views, cfg, dc, tiles, trows, pixels, max_tx, max_rows)) return RAYGS_ERR_INVALID_ARG;
  if (cams[0].mip == RAYGS_MIP_EXACT) return RAYGS_ERR_INVALID_ARG;  // needs the second record buffer

  void *scratch = nullptr;
  s = scratch_for_current_device(&scratch);
  if (s != RAYGS_OK) return s;
  int dev = 0, sms = 0;
  cudaError_t ae = cudaGetDevice(&dev);
  if (ae == cudaSuccess) ae = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (ae != cudaSuccess || sms <= 0) {
    note_cuda_error(ae);
    return RAYGS_ERR_CUDA;
  }

  Work w;
  w.n_views = n_views;
  w.n = n;
  w.tiles = tiles;
  w.trows = trows;
  w.max_tiles_x = max_tx;
  w.max_rows = max_rows;
  w.num_sms = sms;
  w.G = sort_grid(sms);
  w.cfg = cfg;
  if (!fit_scratch(w)) return RAYGS_ERR_CAPACITY;
  w.base = static_cast<char *>(scratch);

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  auto fail = [](cudaError_t e) { note_cuda_error(e); return RAYGS_ERR_CUDA; };
  cudaError_t e = cudaMemcpyAsync(w.base + w.L.cams, dc, sizeof(DevCam) * n_views, cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return fail(e);
  // run_preprocess clears the counters, the only state that must start at zero (the array
  // keeps the previous call's contents)
  if ((e = run_preprocess(w, *scene, st)) != cudaSuccess) return fail(e);
  if ((e = run_bin_sort(w, st)) != cudaSuccess) return fail(e);
  if ((e = run_render(w, rgb, T_final, n_contrib, false, st)) != cudaSuccess) return fail(e);

  // Report an overflow of the tile rows or instances (the image would be incomplete).
  const Counters *ctr = w.at<Counters>(w.L.counters);
  uint32_t overflow = 0;
  if ((e = cudaMemcpyAsync(&overflow, &ctr->overflow, sizeof(overflow), cudaMemcpyDeviceToHost, st)) != cudaSuccess)
    return fail(e);
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return fail(e);
  return overflow ? RAYGS_ERR_CAPACITY : RAYGS_OK;
}

/* Diagnostic, not part of the documented ABI: the capacity a call on a device of `sms` SMs would have
 * in the array (host only), 0 when the batch is refused before any work. */
extern "C" int64_t raygs_debug_noalloc_capacity(const raygs_camera *cams, int32_t n_views, int64_t n,
                                                const raygs_config *cfg, int32_t sms) {
  Work w;
  DevCam dc[RAYGS_MAX_VIEWS];
  int64_t pixels = 0;
  if (!cams || !cfg || n_views < 1 || n_views > RAYGS_MAX_VIEWS || n < 0 || sms < 1) return 0;
  if (!plan_views(cams, n_views, *cfg, dc, w.tiles, w.trows, pixels, w.max_tiles_x, w.max_rows)) return 0;
  w.n_views = n_views;
  w.n = n;
  w.num_sms = sms;
  return fit_scratch(w) ? w.cap : 0;
}
