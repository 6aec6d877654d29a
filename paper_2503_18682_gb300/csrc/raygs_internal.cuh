// Internal declarations shared by the CUDA translation units of the RayGS library.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>

#include "raygs.h"

namespace raygs {

constexpr uint32_t kCulled = 0xFFFFFFFFu;  // depth-key marker of a culled (primitive, view)
constexpr float kLog2e = 1.4426950408889634f;

// Per-view constants as the kernels see them (device copy built by the plan).
struct DevCam {
  float fx, fy, cx, cy;
  float ifx, ify;              // 1/fx, 1/fy
  int W, H;
  float R[9];                  // world -> camera, row-major
  float t[3];
  float near_z;
  int mip;
  float C[3];                  // camera centre in the world frame
  float xmin, xmax, ymin, ymax;  // slopes of the outermost pixel-centre rays
  float fn[4];                 // sqrt(1 + slope^2) of each: norms of the side-plane normals
  int tiles_x, tiles_y;
  int tile_base;               // first global tile id of the view
  int trow_base;               // first global tile row of the view
  long long pix_base;          // first output pixel of the view
};

// 64-byte per-(primitive, view) pixel record consumed by the rasteriser.
//   a = (u_hi, v_hi, u_lo, v_lo)   projected centre in pixels, double-float
//   b = (G00, G01, G10, G11)       y01' = G (px - u) = sqrt(kp) y01, with y01 scaled so that
//                                  y2(centre) = 1; q' = |y01'|^2 = kp |y01|^2
//   c = (h0, h1, kp, c2h)          y2 = 1 + h . (px - u); kp = (c^2-kappa)/kappa;
//                                  c2h = c^2 log2(e) / 2; the support is q' <= y2^2, y2 > 0
//   d = (lo2o, r, g, b)            log2 of the (modulated) opacity; colour
struct __align__(16) Rec {
  float4 a, b, c, d;
};

// Device-side counters (one per workspace).
struct Counters {
  uint32_t n_visible;       // valid (primitive, view) pairs after culling
  uint32_t n_rows_clamped;  // min(tile rows, capacity)
  uint32_t n_inst_clamped;  // min(instances, capacity)
  uint32_t overflow;        // rows or instances exceeded the capacity
  unsigned long long n_rows;
  unsigned long long n_instances;
  unsigned long long n_nonfinite;
  uint32_t n_partials;      // partial-sum slots handed out (plans with the backward)
  uint32_t n_rows_kept;     // support rows with at least one tile
  unsigned long long n_span_rows;  // rows of the pairs whose support is not a bounded ellipse,
  uint32_t n_unbounded;            // and those pairs
  uint32_t n_scan;          // rows of those pairs that have to be tested tile by tile
  uint32_t chunk_rows;      // rows per chunk of the list pass
  uint32_t lists_done;      // CTAs of list_count_kernel that have finished (0 between launches)
  uint32_t longest;                           // longest list of a tile (0 where no classes are kept)
  uint32_t tile_class[16];                    // tiles of each class (see tile_class_of)
};

// Classes of tiles by list length, longest first: the rasteriser takes them in this order (a
// tile with a long list started last would run alone at the end).
constexpr int kTileClasses = 12;
__host__ __device__ constexpr uint32_t tile_class_min(int c) {
  constexpr uint32_t m[kTileClasses] = {4096, 2048, 1024, 768, 512, 384, 256, 192, 128, 64, 16, 0};
  return m[c];
}
__device__ __forceinline__ int tile_class_of(uint32_t len) {
  int c = 0;
#pragma unroll
  for (int k = 0; k < kTileClasses - 1; ++k) c += len < tile_class_min(k) ? 1 : 0;
  return c;
}

// Screen-space support of a (primitive, view), one 32-byte sector for the tile-row pass:
// its tile rectangle (as in the rect array) and the ellipse of pixel centres p with
// (p - c)^T [[a, b], [b, d]] (p - c) <= 1 that holds exactly the rays with D <= kappa (up to
// rounding), det = ad - b^2.  a < 0 marks a support that is not a bounded ellipse in the
// image (or is too ill-conditioned in float32): binning then bounds its rows from the pair's
// record (cx holds, as bits, the pair's first slot among the spans, kCulled when there was no
// room, which only rows beyond the capacity bring about); a = -2 keeps every tile of the rectangle (the
// exact anti-aliasing records hold no conic).
struct __align__(32) Ell {
  uint32_t r0, r1;  // tx0 | ty0 << 16, tx1 | ty1 << 16
  float cx, cy, a, b, d, det;
};

// ---------------------------------------------------------------- double-float helpers
// Error-free transforms (Knuth two-sum, FMA two-product) written with explicitly rounded
// intrinsics so that the compiler cannot contract or reassociate them.
struct df {
  float hi, lo;
};

__device__ __forceinline__ df two_sum(float a, float b) {
  float s = __fadd_rn(a, b);
  float bb = __fsub_rn(s, a);
  float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}

__device__ __forceinline__ df quick_two_sum(float a, float b) {  // requires |a| >= |b|
  float s = __fadd_rn(a, b);
  float e = __fsub_rn(b, __fsub_rn(s, a));
  return {s, e};
}

__device__ __forceinline__ df two_prod(float a, float b) {
  float p = __fmul_rn(a, b);
  float e = __fmaf_rn(a, b, -p);
  return {p, e};
}

__device__ __forceinline__ df df_add(df a, df b) {
  df s = two_sum(a.hi, b.hi);
  float e = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  return quick_two_sum(s.hi, e);
}

__device__ __forceinline__ df df_mul_f(df a, float b) {
  df p = two_prod(a.hi, b);
  float e = __fmaf_rn(a.lo, b, p.lo);
  return quick_two_sum(p.hi, e);
}

// a / b for double-float a, b (one Newton correction; ~44 significant bits).
__device__ __forceinline__ df df_div(df a, df b) {
  float q1 = __fdiv_rn(a.hi, b.hi);
  // r = a - q1 * b
  df p = two_prod(q1, b.hi);
  float r = __fsub_rn(a.hi, p.hi);
  r = __fsub_rn(r, p.lo);
  r = __fadd_rn(r, a.lo);
  r = __fsub_rn(r, __fmul_rn(q1, b.lo));
  float q2 = __fdiv_rn(r, b.hi);
  return quick_two_sum(q1, q2);
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---------------------------------------------------------------- attribute loads
__device__ __forceinline__ float load_attr(const void *base, int64_t idx, int dtype) {
  if (dtype == RAYGS_F16) return __half2float(reinterpret_cast<const __half *>(base)[idx]);
  if (dtype == RAYGS_BF16)
    return __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(base)[idx]);
  return reinterpret_cast<const float *>(base)[idx];
}

inline int dtype_bytes(int dtype) { return dtype == RAYGS_F32 ? 4 : 2; }

// ---------------------------------------------------------------- kernel parameters
struct PrepParams {
  const float *means;
  const void *log_scales;
  const float *quats;
  const void *logits;
  const void *sh;
  int sh_degree, scale_dtype, opacity_dtype, sh_dtype;
  int n;
  int n_views;
  const DevCam *cams;
  float p_min, mip_sigma2, degenerate_ratio;
  int fp64_degenerate;
  int divergence;  // 0: D_ray (Eq. Q_ray); 1: D_gs (Sec. 3.1)
  int tile_w, tile_h;
  uint32_t *depth_key;
  uint2 *rect;
  uint16_t *row_info;   // first tile row (low byte) and tile rows of each pair's rectangle, each saturated at 255
  Ell *ell;
  Rec *rec;
  Rec *recx;            // second half of the exact anti-aliasing record (views with mip = 2)
  Counters *counters;
  uint32_t *span_list;  // pairs whose support is not a bounded ellipse, and room for their rows
  uint32_t span_list_cap, span_cap;
  uint32_t *deg_list;   // (view, primitive) pairs left to the FP64 kernel
  uint32_t *deg_count;
};

struct SortPass {
  const uint32_t *keys_in;
  const uint32_t *vals_in;  // null: the item's index is its value (first depth pass)
  uint32_t *keys_out;
  uint32_t *vals_out;
  uint32_t *index_out;      // the items' indices (the split by view; null otherwise)
  const uint32_t *d_count;  // device item count (nullable: count_max is used)
  uint32_t count_max;
  int shift;
  uint32_t *hist;           // [digits][G]
  uint32_t *digit_total;    // [digits] items of each digit
  int G;
  uint32_t *d_total;        // receives the number of items kept (nullable)
  // The depth sort carries each pair's tile rows: the first pass (row_info: per pair in pair
  // order, first tile row and row count, a byte each, saturated at 255) puts the first tile
  // row in the key's low byte, the digit it has consumed, and min(count, field) into the
  // value's bits above id_bits (a full field or byte means "not known"); the last pass
  // (row_rect set) writes first tile row | (count - 1) << 12 | view << 24 in place of the key
  // and the bare id as the value, taking what is not known from the pair's rectangle.
  // id_bits = 32 leaves no field: every count comes from the rectangle.
  const uint16_t *row_info;
  int id_bits;
  const uint2 *row_rect;
  uint32_t n;               // primitives per view (the last depth pass)
  int n_views;              // views (the split by view)
};

// Support rows of the depth-sorted pairs (rows.cu).
struct PlaceParams {
  const uint32_t *info;        // tile rows of each sorted pair, view by view (see SortPass)
  const uint32_t *pos;         // its position in the depth order (null: one view, the index itself)
  const uint32_t *ids;         // its pair id
  const uint32_t *view_count;  // pairs of each view (null: one view, all of them)
  const Ell *ell;
  const Rec *rec;
  const DevCam *cams;
  Counters *counters;
  int n, n_views, tile_w, tile_h;
  int trows, max_rows;         // tile rows of the batch, and the most of one view
  uint32_t cap;
  uint32_t heads, head_pairs;  // head chunks of a view, at most, and their pairs (see rows.cu)
  uint32_t cp_lo, cp_hi, target;
  const uint32_t *span_list;   // pairs whose support is not a bounded ellipse (see PrepParams)
  uint32_t span_list_cap;
  uint32_t *scan;              // [cap] spans left to be tested tile by tile (in the first half of rows)
  uint32_t *spans;             // per row of those pairs: first tile column | tiles << 16
  uint32_t *cnt1;              // per view, tile row and chunk: rows, then rows of the chunks before
  uint2 *trow_ranges;          // [tile rows] the tile row's range of the row list
  unsigned long long *trow_inst;  // [tile rows] rows, then cleared for the list pass
  uint32_t *chunk_base;        // [tile rows + 1] first chunk of each tile row in the list pass
  uint32_t list_lo, list_hi, list_target, max_chunks;
  uint2 *rows;                 // [cap] the row list: sorted pair position, first tile column | tiles << 16
  // plans with the backward (null otherwise): where each row's instances lie among the partial
  // sums, (chunk, offset in the chunk); the chunks' first slots; per sorted pair its run
  // (first, end, chunk)
  uint2 *row_e;
  uint32_t *e_base;
  uint4 *pair_e;
};

// Instance lists from the support rows listed by tile row, in depth order (lists.cu).
struct ListParams {
  const DevCam *cams;
  int n_views;
  Counters *counters;
  const uint2 *trow_ranges;  // [tile rows] range of the tile row in the row list
  const uint2 *rows;         // the row list (see PlaceParams)
  const uint2 *row_e;
  const uint32_t *e_base;
  uint32_t *inst_e;          // [cap] partial-sum slot of every instance (plans with the backward)
  unsigned long long *trow_inst;  // [tile rows] instances of each tile row, then its first instance
  uint2 *ranges;             // [tiles] instance range of every tile (clamped to cap)
  uint32_t *class_tiles;     // [kTileClasses][tiles] the tiles of each class (nullable)
  int64_t tiles;
  uint32_t *inst;            // [cap] sorted pair position of every instance
  uint32_t cap;
  // Each tile row's rows are cut into chunks (at least one): chunk_base[t] is tile row t's first
  // chunk (chunk_base[trows] the number of chunks), cnt2[chunk][x] the chunk's instances in
  // tile column x.
  const uint32_t *chunk_base;
  uint32_t *cnt2;
  int trows, max_tiles_x;
  uint32_t max_chunks;
};

struct RenderParams {
  const DevCam *cams;
  int n_views;
  const uint2 *ranges;
  const uint32_t *inst_vals;
  const uint32_t *pairs;
  const Rec *rec;
  float t_stop, alpha_max;
  float qmix;  // 1: D_ray fragment formula, D ~ q / (q + r); 0: D_gs, D ~ q (records with h = 0)
  unsigned int *tile_counter;  // [0] next unclaimed item of the persistent rasteriser, [1] CTAs that
                               // have left it; both 0 between launches (the last CTA clears them)
  int n_tiles;
  const uint32_t *class_tiles;  // tiles by class (nullable: tile order)
  const uint32_t *class_count;
  const Counters *counters;
  int slots;                    // CTAs resident at a time (set at the launch)
  const Rec *recx;  // exact anti-aliasing: second half of each record (then rec holds the first)
  float p_min;
  float *rgb;
  float *Tf;
  int *ncontrib;
  // [4]: evaluated and composited (pixel, primitive) pairs, list entries the CTAs staged
  // (consumed instances), (thread, record) iterations with a live pixel
  unsigned long long *eval_counts;
  uint32_t *tile_stop;  // instrumented variant: per tile, list entries staged before every pixel
                        // stopped, or kCulled when the list ran out first (nullable)
};

// The kernels of a pass follow one another in a stream.  Each is launched as a programmatic dependent
// of the one before: it is made ready while that one still runs, its CTAs are placed as the last
// CTAs of that one leave, and wait in await_previous, before they touch memory, until its writes
// are visible.  (Every CTA of every kernel waits, so a kernel's completion implies that of all before
// it.)  That saves about 1.5 us between two kernels: a 64x64 thumbnail of 1,000 primitives 111 -> 77 us,
// a 720p view of 500k primitives 314 -> 263 us, passes of milliseconds unchanged.  Letting the
// next kernel in earlier (launch_dependents at the start of every kernel) gave 96 and 283 us and cost
// the large passes 3 to 6 %: its CTAs take room and are spread unevenly.  A graph under capture
// gets plain edges, which are as fast there.
template <typename... KArgs, typename... Args>
inline cudaError_t launch(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                          const Args &...args) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  const cudaError_t e = cudaStreamIsCapturing(st, &capture);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = capture == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
__device__ __forceinline__ void await_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

constexpr int kMaxTilesX = 4096;  // tiles in one tile row (32768-pixel views at 8-pixel tiles)
constexpr int kGradW = 13;  // per-instance / per-pair gradient partials (see backward.cu)

// What a backward pass has to replay: the lists up to the last composited instance.
struct ReplayPlan {
  uint32_t longest, sum;  // over the tiles
  uint32_t tile_class[kTileClasses];  // tiles of each class, without those that have nothing to replay
  uint32_t fp64_count;  // primitives that param_grads_kernel left to the FP64 kernel
};

struct BackParams {
  const DevCam *cams;
  int n_views;
  const uint2 *ranges;
  const uint32_t *inst_vals;
  const uint32_t *inst_e;  // partial-sum slot of every instance
  const uint32_t *pairs;
  const Rec *rec;
  uint32_t cap;
  float t_stop, alpha_max;
  const float *Tf;
  const int *ncontrib;
  const float *dL_drgb;
  const float *dL_dT;   // nullable
  float *partials;      // [capacity][kGradW] by partial-sum slot
  uint8_t *touched;     // [capacity] slots that hold a partial sum (cleared first; the others are zero)
  unsigned int *tile_counter;  // as in RenderParams
  ReplayPlan *plan;            // cleared first
  uint32_t *class_tiles;       // nullable, the tiles of each class of the plan
  const uint32_t *class_count;
  int n_tiles, slots, num_sms;
};

struct PairGradParams {
  const uint32_t *pairs;
  const uint4 *pair_e;     // per sorted pair: its run of partial sums (first, end, chunk)
  const uint32_t *e_base;
  uint32_t cap;
  const Counters *counters;
  const float *partials;
  const uint8_t *touched;
  float *pg;            // [V*N][kGradW] by pair id, of the pairs with a gradient
  uint8_t *pair_touched;  // [V*N] pairs with a gradient (cleared first)
};

struct ParamGradParams {
  const float *means;
  const void *log_scales;
  const float *quats;
  const void *logits;
  const void *sh;
  int sh_degree, scale_dtype, opacity_dtype, sh_dtype;
  int n, n_views;
  const DevCam *cams;
  float p_min, degenerate_ratio;
  int fp64_degenerate;
  const uint8_t *pair_touched;  // [V*N] pairs with a gradient
  const float *pg;
  float *d_means, *d_log_scales, *d_quats, *d_logits, *d_sh;
  int num_sms;
  uint32_t *fp64_list;   // primitives left to the FP64 kernel (the forward's FP64 pair list,
  uint32_t *fp64_count;  // free by the time of the backward) and their count (zeroed first)
};

// Records e as the thread's last CUDA error (read back by raygs_last_cuda_error).
void note_cuda_error(cudaError_t e);

cudaError_t launch_preprocess(const PrepParams &P, int num_sms, cudaStream_t st);
cudaError_t launch_sort_pass(SortPass p, cudaStream_t st);
bool sort_is_small(uint64_t pairs);  // one kernel for the whole depth sort
cudaError_t launch_sort_small(const SortPass &p, cudaStream_t st);  // row_info, row_rect and d_total set
int sort_blocks(uint64_t items, int grid);  // CTAs of a pass
constexpr int kHeadChunks = 128;  // head chunks of a view in the row pass, where there is room for their counts
uint32_t place_chunk_lo(uint64_t pairs, int max_rows, bool short_chunks);
int place_heads(int max_rows, int64_t trows, bool short_chunks);
uint32_t place_head_pairs(int heads);
uint64_t place_max_chunks(int n_views, uint64_t pairs, uint32_t chunk_lo, int heads);
uint64_t place_max_counts(int n_views, uint64_t pairs, int max_rows, int64_t trows, uint32_t chunk_lo, int heads);
cudaError_t launch_place(PlaceParams P, int num_sms, cudaStream_t st);
constexpr uint32_t kListRowsLo = 512;  // rows of the shortest chunk of the list pass
uint32_t list_rows_short(int max_tiles_x);
uint32_t list_rows_hi(int64_t cap, int max_tiles_x);
uint32_t list_target(int num_sms);
uint64_t list_max_chunks(int64_t trows, int64_t cap, int max_tiles_x, int num_sms, uint32_t rows_lo);
cudaError_t launch_lists(const ListParams &P, int num_sms, cudaStream_t st);
cudaError_t launch_render(const RenderParams &P, int tile_w, int tile_h, int batch_records, int num_sms,
                          bool count, cudaStream_t st);
cudaError_t launch_render_mipx(const RenderParams &P, int tile_w, int tile_h, int num_sms, bool count,
                               cudaStream_t st);
cudaError_t launch_render_backward(const BackParams &P, int tile_w, int tile_h, cudaStream_t st);
cudaError_t launch_pair_grads(const PairGradParams &P, int G, cudaStream_t st);
cudaError_t launch_param_grads(const ParamGradParams &P, cudaStream_t st);
cudaError_t launch_resolve(const float *rgb_hi, const float *T_hi, float *rgb_lo, float *T_lo, int w_lo, int h_lo,
                           int factor, long long base_hi, long long base_lo, cudaStream_t st);

// ---------------------------------------------------------------- workspace
// Byte offsets of every buffer inside one caller-owned (or library-static) workspace.
struct Layout {
  size_t tilectr, tclass, cams, spanl, spans, vpos, counters, evals, tstop, depth, rect, rinfo, ell, rec, recx, s1k[2], s1v[2], cnt1, rows,
      re, ebase, paire, trange, trinst, cbase, ccnt, inst, inste, hist, dtot, ranges, deg, degc, partials, bclass, bplan, ptouch, pg, pgtouch, total;
};

// What a plan keeps besides the buffers that every pass needs.
struct LayoutOptions {
  bool backward = false, mip_exact = false;
  bool tile_order = true;   // the tiles by class (48 bytes per tile): without, they are taken in tile order
  bool tile_stop = true;    // per-tile stop positions (instrumented renders)
  bool bin_once = false;    // one binning per vertex stage: what it reads of that need not outlast it
  int heads = -1;           // head chunks of a view in the row pass (their counts: 4 bytes per tile row each); -1: place_heads
  bool short_chunks = true;        // short chunks of the row pass on tall views (see place_chunk_lo)
  uint32_t list_lo = kListRowsLo;  // rows of the shortest chunk of the list pass (its counts: 4 bytes per tile column)
};

Layout make_layout(int n_views, int64_t n, int64_t tiles, int64_t trows, int64_t cap, int num_sms, int max_tiles_x,
                   int max_rows, const LayoutOptions &opt);

// Workspace bytes per unit of instance capacity (support rows and instances share it), besides the
// column counts of the list pass and the list below.
constexpr size_t kBytesPerCapacity = 8 + 4;
// Room for the pairs whose support is not a bounded ellipse: each has a row at least, so that none is
// left out unless the rows overflow the capacity.  Their rows' spans lie where the instances come
// later, one word per unit of capacity.
constexpr uint32_t span_list_cap(uint64_t pairs, uint64_t cap) { return uint32_t(pairs < cap ? pairs : cap); }

// A bound workspace and the sizes it was laid out for.
struct Work {
  char *base = nullptr;
  Layout L{};
  int n_views = 0;
  int64_t n = 0, tiles = 0, trows = 0, cap = 0;
  int max_tiles_x = 0, max_rows = 0;  // most tile columns and rows of one view
  int G = 0, num_sms = 0, heads = -1;
  bool short_chunks = true;
  uint32_t list_lo = kListRowsLo;
  raygs_config cfg{};
  int s1_final = 0;  // which ping-pong buffer holds the depth-sorted pairs
  template <typename T>
  T *at(size_t off) const { return reinterpret_cast<T *>(base + off); }
};

// Host-side helpers shared by the entry points.
void fill_devcam(const raygs_camera &c, const raygs_config &cfg, DevCam &d);
// Per-view constants and the global tile, tile-row and pixel numbering of a batch of views;
// false when a view is invalid or the batch is too large to number in 31 bits.
bool plan_views(const raygs_camera *cams, int n_views, const raygs_config &cfg, DevCam *dc, int64_t &tiles,
                int64_t &trows, int64_t &pixels, int &max_tiles_x, int &max_rows);
bool config_valid(const raygs_config &cfg);
bool camera_valid(const raygs_camera &c);
raygs_status scene_valid(const raygs_scene *s, int64_t n);

int sort_grid(int num_sms);
cudaError_t run_preprocess(Work &w, const raygs_scene &scene, cudaStream_t st);
cudaError_t run_bin_sort(Work &w, cudaStream_t st);
cudaError_t run_render(const Work &w, float *rgb, float *T_final, int32_t *n_contrib, bool count,
                       cudaStream_t st);
cudaError_t run_backward(const Work &w, const raygs_scene &scene, const float *T_final, const int32_t *n_contrib,
                         const float *dL_drgb, const float *dL_dT, const raygs_grads &grads, cudaStream_t st);

}  // namespace raygs
