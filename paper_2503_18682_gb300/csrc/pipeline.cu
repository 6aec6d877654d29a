// Workspace layout and the order of kernel launches of the three hot-path stages, shared
// by the plan API (caller-owned workspace) and the allocation-free entry point.
#include <cmath>

#include <algorithm>

#include "raygs_internal.cuh"

namespace raygs {

namespace {
size_t up256(size_t x) { return (x + 255) / 256 * 256; }
}  // namespace

void fill_devcam(const raygs_camera &c, const raygs_config &cfg, DevCam &d) {
  d = DevCam{};
  d.fx = c.fx; d.fy = c.fy; d.cx = c.cx; d.cy = c.cy;
  d.ifx = float(1.0 / double(c.fx));
  d.ify = float(1.0 / double(c.fy));
  d.W = c.width; d.H = c.height;
  for (int i = 0; i < 9; ++i) d.R[i] = c.R[i];
  for (int i = 0; i < 3; ++i) d.t[i] = c.t[i];
  d.near_z = c.near_z;
  d.mip = c.mip;
  for (int k = 0; k < 3; ++k)
    d.C[k] = float(-(double(c.R[k]) * c.t[0] + double(c.R[3 + k]) * c.t[1] + double(c.R[6 + k]) * c.t[2]));
  d.xmin = float((0.5 - double(c.cx)) / double(c.fx));
  d.xmax = float((double(c.width) - 0.5 - double(c.cx)) / double(c.fx));
  d.ymin = float((0.5 - double(c.cy)) / double(c.fy));
  d.ymax = float((double(c.height) - 0.5 - double(c.cy)) / double(c.fy));
  const float sl[4] = {d.xmin, d.xmax, d.ymin, d.ymax};
  for (int k = 0; k < 4; ++k) d.fn[k] = float(std::sqrt(1.0 + double(sl[k]) * double(sl[k])));
  d.tiles_x = (c.width + cfg.tile_w - 1) / cfg.tile_w;
  d.tiles_y = (c.height + cfg.tile_h - 1) / cfg.tile_h;
}

bool config_valid(const raygs_config &cfg) {
  const bool tile_ok = (cfg.tile_w == 16 && cfg.tile_h == 16) || (cfg.tile_w == 16 && cfg.tile_h == 8) ||
                       (cfg.tile_w == 32 && cfg.tile_h == 16) || (cfg.tile_w == 8 && cfg.tile_h == 8);
  return tile_ok && cfg.p_min > 0.f && cfg.p_min < 1.f && cfg.t_stop >= 0.f && cfg.t_stop < 1.f &&
         cfg.alpha_max > 0.f && cfg.alpha_max < 1.f && cfg.mip_sigma2 >= 0.f && cfg.degenerate_ratio > 1.f &&
         cfg.fp64_degenerate >= 0 && cfg.fp64_degenerate <= 2 && (cfg.enable_backward == 0 || cfg.enable_backward == 1) &&
         (cfg.batch_records == 1 || cfg.batch_records == 2) && (cfg.divergence == 0 || cfg.divergence == 1) &&
         !(cfg.divergence == 1 && cfg.enable_backward);
}

bool camera_valid(const raygs_camera &c) {
  return c.width >= 1 && c.height >= 1 && c.width <= 32768 && c.height <= 32768 && c.fx > 0.f && c.fy > 0.f &&
         std::isfinite(c.fx) && std::isfinite(c.fy) && std::isfinite(c.cx) && std::isfinite(c.cy) &&
         c.near_z > 0.f && c.mip >= RAYGS_MIP_OFF && c.mip <= RAYGS_MIP_EXACT;
}

raygs_status scene_valid(const raygs_scene *s, int64_t n) {
  if (!s || s->n != n) return RAYGS_ERR_INVALID_ARG;
  if (s->sh_degree < 0 || s->sh_degree > 3) return RAYGS_ERR_INVALID_ARG;
  auto dt_ok = [](int d, bool allow_bf16) {
    return d == RAYGS_F32 || d == RAYGS_F16 || (allow_bf16 && d == RAYGS_BF16);
  };
  if (!dt_ok(s->scale_dtype, true) || !dt_ok(s->opacity_dtype, false) || !dt_ok(s->sh_dtype, true))
    return RAYGS_ERR_INVALID_ARG;
  auto a16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  if (s->n > 0) {
    if (!s->means || !s->log_scales || !s->quats || !s->opacity_logits || !s->sh) return RAYGS_ERR_INVALID_ARG;
    if (!a16(s->means) || !a16(s->log_scales) || !a16(s->quats) || !a16(s->opacity_logits) || !a16(s->sh))
      return RAYGS_ERR_INVALID_ARG;
  }
  return RAYGS_OK;
}

int sort_grid(int num_sms) {
  int g = 4 * num_sms;
  return g > 1024 ? 1024 : (g < 1 ? 1 : g);
}

Layout make_layout(int n_views, int64_t n, int64_t tiles, int64_t trows, int64_t cap, int num_sms, int max_tiles_x,
                   int max_rows, const LayoutOptions &opt) {
  const bool backward = opt.backward;
  Layout L{};
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t r = o; o = up256(o + bytes); return r; };
  const size_t VN = size_t(n_views) * size_t(n);
  const size_t C = size_t(cap);
  L.cams = take(sizeof(DevCam) * size_t(n_views));
  L.counters = take(sizeof(Counters) + 16);  // and the rasteriser's tile counter
  L.tilectr = L.counters + sizeof(Counters);
  L.degc = L.tilectr + 8;  // cleared with the counters
  L.evals = take(4 * sizeof(unsigned long long));
  L.depth = take(4 * VN);
  L.rect = take(8 * VN);
  L.rinfo = take(2 * VN);
  L.ell = take(sizeof(Ell) * VN);
  L.rec = take(sizeof(Rec) * VN);
  L.recx = opt.mip_exact ? take(sizeof(Rec) * VN) : 0;
  for (int i = 0; i < 2; ++i) { L.s1k[i] = take(4 * VN); L.s1v[i] = take(4 * VN); }
  L.vpos = n_views > 1 ? take(4 * VN) : 0;
  const uint32_t chunk_lo = place_chunk_lo(VN, max_rows, opt.short_chunks);
  const int heads = opt.heads < 0 ? place_heads(max_rows, trows, opt.short_chunks) : opt.heads;
  const uint64_t pchunks = place_max_chunks(n_views, VN, chunk_lo, heads);
  L.cnt1 = take(4 * size_t(place_max_counts(n_views, VN, max_rows, trows, chunk_lo, heads)) + 16);
  // per unit of capacity: kBytesPerCapacity bytes
  L.rows = take(8 * C + 16);
  L.spanl = opt.bin_once ? L.rows + 4 * C : take(4 * size_t(span_list_cap(VN, C)));
  L.inst = take(4 * C + 16);
  L.spans = L.inst;  // read by the row pass, before the lists are written
  L.re = backward ? take(8 * C + 16) : 0;
  L.inste = backward ? take(4 * C + 16) : 0;
  L.ebase = backward ? take(4 * pchunks + 16) : 0;
  L.paire = backward ? take(16 * VN + 16) : 0;
  L.trange = take(8 * size_t(trows) + 16);
  L.trinst = take(8 * size_t(trows) + 16);
  L.cbase = take(4 * size_t(trows + 1) + 16);
  L.ccnt = take(4 * size_t(list_max_chunks(trows, cap, max_tiles_x, num_sms, opt.list_lo)) * size_t(max_tiles_x) + 16);
  L.hist = take(4 * 256 * size_t(sort_blocks(VN, sort_grid(num_sms))));
  L.dtot = take(4 * 256);
  L.ranges = take(8 * size_t(tiles));
  L.tclass = opt.tile_order ? take(4 * size_t(kTileClasses) * size_t(tiles) + 16) : 0;
  L.tstop = opt.tile_stop ? take(4 * size_t(tiles) + 16) : 0;
  L.deg = L.s1k[0];  // the FP64 lists of the vertex stage and of the backward: free then
  L.partials = backward ? take(4 * kGradW * C + 16) : 0;
  L.bclass = backward ? take(4 * size_t(kTileClasses) * size_t(tiles) + 16) : 0;
  L.bplan = backward ? take(sizeof(ReplayPlan)) : 0;
  L.ptouch = backward ? take(C + 16) : 0;
  L.pgtouch = backward ? take(VN + 16) : 0;
  L.pg = backward ? take(4 * kGradW * VN + 16) : 0;
  L.total = o;
  return L;
}

bool plan_views(const raygs_camera *cams, int n_views, const raygs_config &cfg, DevCam *dc, int64_t &tiles,
                int64_t &trows, int64_t &pixels, int &max_tiles_x, int &max_rows) {
  tiles = 0; trows = 0; pixels = 0; max_tiles_x = 0; max_rows = 0;
  for (int v = 0; v < n_views; ++v) {
    if (!camera_valid(cams[v])) return false;
    if (cfg.divergence == 1 && cams[v].mip) return false;  // Eq. mip is a RayGS term
    // the exact anti-aliasing uses its own record and rasteriser for the whole batch
    if ((cams[v].mip == RAYGS_MIP_EXACT) != (cams[0].mip == RAYGS_MIP_EXACT)) return false;
    fill_devcam(cams[v], cfg, dc[v]);
    if (dc[v].tiles_x > kMaxTilesX) return false;
    dc[v].tile_base = int(tiles);
    dc[v].trow_base = int(trows);
    dc[v].pix_base = pixels;
    tiles += int64_t(dc[v].tiles_x) * dc[v].tiles_y;
    trows += dc[v].tiles_y;
    pixels += int64_t(cams[v].width) * cams[v].height;
    if (dc[v].tiles_x > max_tiles_x) max_tiles_x = dc[v].tiles_x;
    if (dc[v].tiles_y > max_rows) max_rows = dc[v].tiles_y;
    if (tiles >= (int64_t(1) << 31)) return false;
  }
  return true;
}

cudaError_t run_preprocess(Work &w, const raygs_scene &scene, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(w.base + w.L.counters, 0, sizeof(Counters) + 16, st);
  if (e != cudaSuccess) return e;
  PrepParams P{};
  P.means = scene.means;
  P.log_scales = scene.log_scales;
  P.quats = scene.quats;
  P.logits = scene.opacity_logits;
  P.sh = scene.sh;
  P.sh_degree = scene.sh_degree;
  P.scale_dtype = scene.scale_dtype;
  P.opacity_dtype = scene.opacity_dtype;
  P.sh_dtype = scene.sh_dtype;
  P.n = int(w.n);
  P.n_views = w.n_views;
  P.cams = w.at<DevCam>(w.L.cams);
  P.p_min = w.cfg.p_min;
  P.mip_sigma2 = w.cfg.mip_sigma2;
  P.degenerate_ratio = w.cfg.degenerate_ratio;
  P.fp64_degenerate = w.cfg.fp64_degenerate;
  P.divergence = w.cfg.divergence;
  P.tile_w = w.cfg.tile_w;
  P.tile_h = w.cfg.tile_h;
  P.depth_key = w.at<uint32_t>(w.L.depth);
  P.rect = w.at<uint2>(w.L.rect);
  P.row_info = w.at<uint16_t>(w.L.rinfo);
  P.ell = w.at<Ell>(w.L.ell);
  P.rec = w.at<Rec>(w.L.rec);
  P.recx = w.L.recx ? w.at<Rec>(w.L.recx) : nullptr;
  P.counters = w.at<Counters>(w.L.counters);
  P.span_list = w.at<uint32_t>(w.L.spanl);
  P.span_list_cap = span_list_cap(uint64_t(w.n_views) * uint64_t(w.n), uint64_t(w.cap));
  P.span_cap = uint32_t(w.cap);
  P.deg_list = w.at<uint32_t>(w.L.deg);
  P.deg_count = w.at<uint32_t>(w.L.degc);
  return launch_preprocess(P, w.num_sms, st);
}

cudaError_t run_bin_sort(Work &w, cudaStream_t st) {
  Counters *ctr = w.at<Counters>(w.L.counters);
  const uint32_t VN = uint32_t(size_t(w.n_views) * size_t(w.n));
  const uint32_t cap = uint32_t(w.cap);
  cudaError_t e;
  SortPass base{};
  base.hist = w.at<uint32_t>(w.L.hist);
  base.digit_total = w.at<uint32_t>(w.L.dtot);
  base.G = w.G;
  base.count_max = VN;
  base.n = uint32_t(w.n);
  base.n_views = w.n_views;
  // 1. depth sort of the visible pairs: 4 passes of 8 bits over the float32 key, which carry
  // each pair's tile rows (the values' bits above those of the largest id, and the key's
  // consumed digit)
  base.id_bits = 1;
  while (base.id_bits < 32 && (uint64_t(1) << base.id_bits) < uint64_t(VN)) ++base.id_bits;
  int cur = 0;
  const bool small = sort_is_small(VN);
  if (small) {
    SortPass sp = base;
    sp.keys_in = w.at<uint32_t>(w.L.depth);
    sp.keys_out = w.at<uint32_t>(w.L.s1k[cur]);
    sp.vals_out = w.at<uint32_t>(w.L.s1v[cur]);
    sp.d_total = &ctr->n_visible;
    sp.row_info = w.at<uint16_t>(w.L.rinfo);
    sp.row_rect = w.at<uint2>(w.L.rect);
    if ((e = launch_sort_small(sp, st)) != cudaSuccess) return e;
  }
  for (int pass = 0; pass < (small ? 0 : 4); ++pass) {
    SortPass sp = base;
    sp.keys_in = w.at<uint32_t>(pass == 0 ? w.L.depth : w.L.s1k[cur]);
    sp.vals_in = pass == 0 ? nullptr : w.at<uint32_t>(w.L.s1v[cur]);
    const int dst = pass == 0 ? 0 : 1 - cur;
    sp.keys_out = w.at<uint32_t>(w.L.s1k[dst]);
    sp.vals_out = w.at<uint32_t>(w.L.s1v[dst]);
    sp.d_count = pass == 0 ? nullptr : &ctr->n_visible;
    sp.shift = 8 * pass;
    sp.d_total = pass == 0 ? &ctr->n_visible : nullptr;
    sp.row_info = pass == 0 ? w.at<uint16_t>(w.L.rinfo) : nullptr;
    sp.row_rect = pass == 3 ? w.at<uint2>(w.L.rect) : nullptr;
    if ((e = launch_sort_pass(sp, st)) != cudaSuccess) return e;
    cur = dst;
  }
  w.s1_final = cur;
  // 2. several views: the pairs view by view (stable), with their positions in the depth order;
  // the other ping-pong buffer takes the result, the depth order stays
  const bool split = w.n_views > 1;
  if (split) {
    SortPass sp = base;
    sp.keys_in = w.at<uint32_t>(w.L.s1k[cur]);
    sp.keys_out = w.at<uint32_t>(w.L.s1k[1 - cur]);
    sp.vals_in = w.at<uint32_t>(w.L.s1v[cur]);
    sp.vals_out = w.at<uint32_t>(w.L.s1v[1 - cur]);
    sp.index_out = w.at<uint32_t>(w.L.vpos);
    sp.d_count = &ctr->n_visible;
    sp.shift = 24;
    if ((e = launch_sort_pass(sp, st)) != cudaSuccess) return e;
  }
  // 3. support rows into per-tile-row lists
  PlaceParams R{};
  R.info = w.at<uint32_t>(w.L.s1k[split ? 1 - cur : cur]);
  R.pos = split ? w.at<uint32_t>(w.L.vpos) : nullptr;
  R.ids = w.at<uint32_t>(w.L.s1v[split ? 1 - cur : cur]);
  R.view_count = split ? base.digit_total : nullptr;
  R.ell = w.at<Ell>(w.L.ell);
  R.rec = w.at<Rec>(w.L.rec);
  R.cams = w.at<DevCam>(w.L.cams);
  R.counters = ctr;
  R.n = int(w.n);
  R.n_views = w.n_views;
  R.tile_w = w.cfg.tile_w;
  R.tile_h = w.cfg.tile_h;
  R.trows = int(w.trows);
  R.max_rows = w.max_rows;
  R.cap = cap;
  R.heads = uint32_t(w.heads < 0 ? place_heads(w.max_rows, w.trows, w.short_chunks) : w.heads);
  R.cp_lo = place_chunk_lo(VN, w.max_rows, w.short_chunks);
  R.span_list = w.at<uint32_t>(w.L.spanl);
  R.span_list_cap = span_list_cap(VN, cap);
  R.spans = w.at<uint32_t>(w.L.spans);
  R.scan = w.at<uint32_t>(w.L.rows);
  R.cnt1 = w.at<uint32_t>(w.L.cnt1);
  R.trow_ranges = w.at<uint2>(w.L.trange);
  R.trow_inst = w.at<unsigned long long>(w.L.trinst);
  R.rows = w.at<uint2>(w.L.rows);
  R.chunk_base = w.at<uint32_t>(w.L.cbase);
  R.list_lo = w.list_lo;
  R.list_hi = list_rows_hi(w.cap, w.max_tiles_x);
  R.list_target = list_target(w.num_sms);
  R.max_chunks = uint32_t(list_max_chunks(w.trows, w.cap, w.max_tiles_x, w.num_sms, w.list_lo));
  const bool backward = w.cfg.enable_backward != 0;
  R.row_e = backward ? w.at<uint2>(w.L.re) : nullptr;
  R.e_base = backward ? w.at<uint32_t>(w.L.ebase) : nullptr;
  R.pair_e = backward ? w.at<uint4>(w.L.paire) : nullptr;
  if ((e = launch_place(R, w.num_sms, st)) != cudaSuccess) return e;
  // 4. instances per tile, tile offsets, lists
  ListParams X{};
  X.cams = R.cams;
  X.n_views = w.n_views;
  X.counters = ctr;
  X.trow_ranges = R.trow_ranges;
  X.rows = R.rows;
  X.row_e = R.row_e;
  X.e_base = R.e_base;
  X.inst_e = backward ? w.at<uint32_t>(w.L.inste) : nullptr;
  X.trow_inst = R.trow_inst;
  X.ranges = w.at<uint2>(w.L.ranges);
  X.class_tiles = w.L.tclass ? w.at<uint32_t>(w.L.tclass) : nullptr;
  X.tiles = w.tiles;
  X.inst = w.at<uint32_t>(w.L.inst);
  X.cap = cap;
  X.chunk_base = R.chunk_base;
  X.cnt2 = w.at<uint32_t>(w.L.ccnt);
  X.trows = int(w.trows);
  X.max_tiles_x = w.max_tiles_x;
  X.max_chunks = R.max_chunks;
  return launch_lists(X, w.num_sms, st);
}

cudaError_t run_render(const Work &w, float *rgb, float *T_final, int32_t *n_contrib, bool count,
                       cudaStream_t st) {
  RenderParams P{};
  P.cams = w.at<DevCam>(w.L.cams);
  P.n_views = w.n_views;
  P.ranges = w.at<uint2>(w.L.ranges);
  P.inst_vals = w.at<uint32_t>(w.L.inst);
  P.pairs = w.at<uint32_t>(w.L.s1v[w.s1_final]);
  P.rec = w.at<Rec>(w.L.rec);
  P.t_stop = w.cfg.t_stop;
  P.alpha_max = w.cfg.alpha_max;
  P.qmix = w.cfg.divergence == 1 ? 0.f : 1.f;
  P.recx = w.L.recx ? w.at<Rec>(w.L.recx) : nullptr;
  P.p_min = w.cfg.p_min;
  P.rgb = rgb;
  P.Tf = T_final;
  P.ncontrib = n_contrib;
  P.eval_counts = w.at<unsigned long long>(w.L.evals);
  P.tile_stop = count ? w.at<uint32_t>(w.L.tstop) : nullptr;
  if (count) {
    cudaError_t e = cudaMemsetAsync(P.eval_counts, 0, 4 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
  }
  if (w.tiles == 0) return cudaSuccess;
  P.tile_counter = w.at<unsigned int>(w.L.tilectr);
  P.n_tiles = int(w.tiles);
  P.class_tiles = w.L.tclass ? w.at<uint32_t>(w.L.tclass) : nullptr;
  P.counters = w.at<Counters>(w.L.counters);
  P.class_count = P.counters->tile_class;
  if (P.recx) return launch_render_mipx(P, w.cfg.tile_w, w.cfg.tile_h, w.num_sms, count, st);
  return launch_render(P, w.cfg.tile_w, w.cfg.tile_h, w.cfg.batch_records, w.num_sms, count, st);
}

cudaError_t run_backward(const Work &w, const raygs_scene &scene, const float *T_final, const int32_t *n_contrib,
                         const float *dL_drgb, const float *dL_dT, const raygs_grads &grads, cudaStream_t st) {
  BackParams B{};
  B.cams = w.at<DevCam>(w.L.cams);
  B.n_views = w.n_views;
  B.ranges = w.at<uint2>(w.L.ranges);
  B.inst_vals = w.at<uint32_t>(w.L.inst);
  B.pairs = w.at<uint32_t>(w.L.s1v[w.s1_final]);
  B.rec = w.at<Rec>(w.L.rec);
  B.inst_e = w.at<uint32_t>(w.L.inste);
  B.cap = uint32_t(w.cap);
  B.t_stop = w.cfg.t_stop;
  B.alpha_max = w.cfg.alpha_max;
  B.Tf = T_final;
  B.ncontrib = n_contrib;
  B.dL_drgb = dL_drgb;
  B.dL_dT = dL_dT;
  B.partials = w.at<float>(w.L.partials);
  B.touched = w.at<uint8_t>(w.L.ptouch);
  B.tile_counter = w.at<unsigned int>(w.L.tilectr);
  B.n_tiles = int(w.tiles);
  B.plan = w.at<ReplayPlan>(w.L.bplan);
  B.class_tiles = w.at<uint32_t>(w.L.bclass);
  B.class_count = B.plan->tile_class;
  B.num_sms = w.num_sms > 0 ? w.num_sms : 1;
  uint8_t *pair_touched = w.at<uint8_t>(w.L.pgtouch);
  // the plan, touched and pair_touched lie behind one another: one clear
  cudaError_t e = cudaMemsetAsync(B.plan, 0, w.L.pgtouch - w.L.bplan + size_t(w.n_views) * size_t(w.n), st);
  if (e != cudaSuccess) return e;
  if ((e = launch_render_backward(B, w.cfg.tile_w, w.cfg.tile_h, st)) != cudaSuccess) return e;
  PairGradParams Q{};
  Q.pairs = B.pairs;
  Q.pair_e = w.at<uint4>(w.L.paire);
  Q.e_base = w.at<uint32_t>(w.L.ebase);
  Q.cap = B.cap;
  Q.counters = w.at<Counters>(w.L.counters);
  Q.partials = B.partials;
  Q.touched = B.touched;
  Q.pg = w.at<float>(w.L.pg);
  Q.pair_touched = pair_touched;
  if ((e = launch_pair_grads(Q, w.G, st)) != cudaSuccess) return e;
  ParamGradParams R{};
  R.means = scene.means;
  R.log_scales = scene.log_scales;
  R.quats = scene.quats;
  R.logits = scene.opacity_logits;
  R.sh = scene.sh;
  R.sh_degree = scene.sh_degree;
  R.scale_dtype = scene.scale_dtype;
  R.opacity_dtype = scene.opacity_dtype;
  R.sh_dtype = scene.sh_dtype;
  R.n = int(w.n);
  R.n_views = w.n_views;
  R.cams = B.cams;
  R.p_min = w.cfg.p_min;
  R.degenerate_ratio = w.cfg.degenerate_ratio;
  R.fp64_degenerate = w.cfg.fp64_degenerate;
  R.pair_touched = pair_touched;
  R.pg = Q.pg;
  R.d_means = grads.d_means;
  R.d_log_scales = grads.d_log_scales;
  R.d_quats = grads.d_quats;
  R.d_logits = grads.d_opacity_logits;
  R.d_sh = grads.d_sh;
  R.num_sms = w.num_sms;
  R.fp64_list = w.at<uint32_t>(w.L.deg);
  R.fp64_count = &B.plan->fp64_count;
  return launch_param_grads(R, st);
}

}  // namespace raygs
