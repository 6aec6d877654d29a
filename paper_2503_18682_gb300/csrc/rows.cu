// Support rows of the depth-sorted pairs, placed straight into per-tile-row lists in depth
// order: each pair covers the tile rows of its screen rectangle, and each of those rows gets
// the run of tiles whose pixel centres can meet the pair's support (the band of a bounded
// ellipse, or an exact conic test).
//
// The pairs come view by view (depth order inside a view), so that a chunk of them meets
// only its view's tile rows (138 on a 2064 x 2208 eye, not the batch's 1,522) and the 32-byte
// support sectors gathered together belong to one view.
//   pair_count_kernel  per chunk and tile row, the chunk's rows (from the pairs' tile-row
//                      ranges alone, which ride through the depth sort), and the spans of
//                      the few pairs whose support is not a bounded ellipse
//   row_base_kernel    per tile row, the exclusive scan of its chunks' counts
//   trow_plan_kernel   the tile rows' ranges, the row total and the capacity check
//   place_kernel       the rows themselves
// Against writing the rows in pair order and sorting them by tile row (two radix passes of
// keyed rows): binning of the 3M-primitive stereo batch 3.17 against 4.0 ms.
#include <algorithm>

#include "bins.cuh"

namespace raygs {

// ------------------------------------------------------------ support of one tile row

// Pixel-centre columns of the band ya <= y <= yb (pixel-centre rows) inside the ellipse.
// The right boundary x_r(y) is concave with its maximum at the rightmost point of the
// ellipse, the left one convex: clamping that point's y into the band gives the extremes.
struct Band {
  float cx, cy, a, b, det, hy, ydx;
};
__device__ __forceinline__ Band band_of(const Ell &e) {
  Band q;
  const float rho = 1.001f;
  q.cx = e.cx; q.cy = e.cy; q.a = e.a; q.b = e.b; q.det = e.det;
  q.hy = sqrtf(rho * e.a / e.det);
  const float hx = sqrtf(rho * e.d / e.det);
  q.ydx = -e.b * hx / e.d;  // y offset of the rightmost point
  return q;
}
__device__ __forceinline__ bool ellipse_band(const Band &e, float ya, float yb, float &xa, float &xb) {
  const float rho = 1.001f;
  const float lo = fmaxf(ya - e.cy, -e.hy), hi = fminf(yb - e.cy, e.hy);
  if (lo > hi) return false;
  const float yr = fminf(fmaxf(e.ydx, lo), hi), yl = fminf(fmaxf(-e.ydx, lo), hi);
  const float xr = (-e.b * yr + sqrtf(fmaxf(e.a * rho - e.det * yr * yr, 0.f))) / e.a;
  const float xl = (-e.b * yl - sqrtf(fmaxf(e.a * rho - e.det * yl * yl, 0.f))) / e.a;
  xa = e.cx + xl;
  xb = e.cx + xr;
  return true;
}

// Supports that are not a bounded ellipse (the primitive's cone of rays reaches the
// camera plane, or the ellipse is too ill-conditioned in float32) are still convex: the
// image of one nappe of an elliptic cone cut by the plane z = 1.  Within a band of pixel
// rows their pixels therefore occupy one contiguous run of tiles, whose ends are found by
// bisection with a vertical-line test.

// Does the segment delta(t) = P + t E, t in [0, 1] (pixel offsets from the projected
// centre) meet the support |G delta|^2 <= y2^2, y2 = 1 + h.delta > 0 (the record's G carries
// sqrt(kp))?  Along the segment y01' = a + t b and y2 = al + t be, so f = |y01'|^2 - y2^2 is a
// quadratic in t;
// its minimum over the part where y2 > 0 is compared with a margin of 1e-4 of the
// magnitude of its terms, far above float32 rounding: the answer errs only towards yes.
// t_at receives the parameter of that minimum.
__device__ __forceinline__ bool segment_meets_support(const Rec &r, float Px, float Py, float Ex, float Ey,
                                                      float *t_at = nullptr) {
  const float kp = 1.f;
  const float a0 = fmaf(r.b.x, Px, r.b.y * Py), a1 = fmaf(r.b.z, Px, r.b.w * Py);
  const float b0 = fmaf(r.b.x, Ex, r.b.y * Ey), b1 = fmaf(r.b.z, Ex, r.b.w * Ey);
  const float al = fmaf(r.c.x, Px, fmaf(r.c.y, Py, 1.f)), be = fmaf(r.c.x, Ex, r.c.y * Ey);
  const float slack = 1e-5f * (fabsf(al) + fabsf(be)) + 1e-6f;
  float t0 = 0.f, t1 = 1.f;
  if (be > 0.f) t0 = fmaxf(t0, (-slack - al) / be);
  else if (be < 0.f) t1 = fminf(t1, (-slack - al) / be);
  else if (al < -slack) return false;
  if (!(t0 <= t1)) return false;
  const float qa = fmaf(a0, a0, a1 * a1), qb = fmaf(b0, b0, b1 * b1), qab = fmaf(a0, b0, a1 * b1);
  const float A = fmaf(kp, qb, -be * be);
  const float Bh = fmaf(kp, qab, -al * be);
  const float Cc = fmaf(kp, qa, -al * al);
  const float margin = 1e-4f * (2.f * fmaf(kp, qa, al * al) + 2.f * fmaf(kp, qb, be * be)) + 1e-6f;
  const float f0 = fmaf(fmaf(A, t0, 2.f * Bh), t0, Cc), f1 = fmaf(fmaf(A, t1, 2.f * Bh), t1, Cc);
  float m = f0, tm = t0;
  if (f1 < m) { m = f1; tm = t1; }
  if (A > 0.f) {
    const float tv = -Bh / A;
    if (tv > t0 && tv < t1) {
      const float fv = fmaf(Bh, tv, Cc);
      if (fv < m) { m = fv; tm = tv; }
    }
  }
  if (t_at) *t_at = tm;
  return m <= margin;
}

// Can the pixel centres of the rectangle [dxa, dxb] x [dya, dyb] (offsets from the projected
// centre) meet the support?  For a convex support: the rectangle holds the projected centre,
// or one of its edges meets the support.
__device__ __forceinline__ bool tile_meets_support(const Rec &r, float dxa, float dxb, float dya, float dyb) {
  return (dxa <= 0.f && dxb >= 0.f && dya <= 0.f && dyb >= 0.f) ||
         segment_meets_support(r, dxa, dya, 0.f, dyb - dya) || segment_meets_support(r, dxb, dya, 0.f, dyb - dya) ||
         segment_meets_support(r, dxa, dya, dxb - dxa, 0.f) || segment_meets_support(r, dxa, dyb, dxb - dxa, 0.f);
}

// First and last tile column in [tx0, tx1] whose pixel centres in rows [ya, yb] can meet
// the support: 1, or 0 if none, or -1 when the tiles have to be tested one by one
// (scan_tile_span).  A point of the support inside the band is found on the
// band's boundary or is the projected centre itself (a convex set that meets a rectangle
// but not its boundary lies inside it).  Left of that point, tile t meets the support
// exactly when the vertical line through its last pixel-centre column does (the support's
// columns within the band form an interval), and symmetrically on the right.
__device__ __noinline__ int support_tile_span(const Rec &r, const DevCam &cam, int tile_w, float ya, float yb, int tx0, int tx1,
                                  int &first, int &last) {
  const float ux = r.a.x, uy = r.a.y, lx = r.a.z, ly = r.a.w;
  const float dya = (ya - uy) - ly, dyb = (yb - uy) - ly;
  auto col_dx = [&](int px_centre_times2) {  // pixel-centre column (2x, exact) as an offset
    return (0.5f * float(px_centre_times2) - ux) - lx;
  };
  auto left_col = [&](int tx) { return col_dx(2 * tx * tile_w + 1); };
  auto right_col = [&](int tx) { return col_dx(2 * min((tx + 1) * tile_w, cam.W) - 1); };
  auto vert = [&](float dx) { return segment_meets_support(r, dx, dya, 0.f, dyb - dya); };
  const float dxL = left_col(tx0), dxR = right_col(tx1);
  // a tile that holds a point of the support (any tile at least as wide as that point's
  // pixel column is a conservative choice)
  int tstar = -1;
  float t;
  if (vert(dxL)) {
    tstar = tx0;
  } else if (vert(dxR)) {
    tstar = tx1;
  } else {
    float cx = 0.f;
    bool inside = dya <= 0.f && dyb >= 0.f && dxL <= 0.f && dxR >= 0.f;
    if (!inside && segment_meets_support(r, dxL, dya, dxR - dxL, 0.f, &t)) { inside = true; cx = fmaf(t, dxR - dxL, dxL); }
    if (!inside && segment_meets_support(r, dxL, dyb, dxR - dxL, 0.f, &t)) { inside = true; cx = fmaf(t, dxR - dxL, dxL); }
    if (!inside) return 0;
    // the minimum along a long horizontal segment carries a wide margin: confirm the point
    // with the (short) vertical test, else the row is scanned tile by tile
    if (!vert(cx)) return -1;
    const float px = (cx + lx) + ux;  // pixel x of the point
    tstar = min(max(int(floorf(px / float(tile_w))), tx0), tx1);
  }
  int lo = tx0, hi = tstar;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (vert(right_col(mid))) hi = mid; else lo = mid + 1;
  }
  first = lo;
  lo = tstar; hi = tx1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (vert(left_col(mid))) lo = mid; else hi = mid - 1;
  }
  last = lo;
  return 1;
}

// The same span by testing the row's tiles, 32 at a time: the whole warp works on one row
// (every argument is the warp's).  Nearly every row that comes here turns out empty; tested by
// one lane, tile after tile, a row of 160 tiles took 70 us and was the length of the binning
// of a frame with a single such primitive.
__device__ __noinline__ bool scan_tile_span(const Rec &r, const DevCam &cam, int tile_w, float ya, float yb, int tx0,
                                            int tx1, int &first, int &last) {
  const int lane = threadIdx.x & 31;
  const float dya = (ya - r.a.y) - r.a.w, dyb = (yb - r.a.y) - r.a.w;
  auto meets = [&](int tx) {
    const float dxa = (0.5f * float(2 * tx * tile_w + 1) - r.a.x) - r.a.z;
    const float dxb = (0.5f * float(2 * min((tx + 1) * tile_w, cam.W) - 1) - r.a.x) - r.a.z;
    return tx <= tx1 && tile_meets_support(r, dxa, dxb, dya, dyb);
  };
  first = tx1 + 1;
  for (int t = tx0; t <= tx1; t += 32) {
    const uint32_t hit = __ballot_sync(0xffffffffu, meets(t + lane));
    if (hit) {
      first = t + __ffs(hit) - 1;
      last = t + 31 - __clz(hit);
      for (t += 32; t <= tx1; t += 32) {
        const uint32_t more = __ballot_sync(0xffffffffu, meets(t + lane));
        if (more) last = t + 31 - __clz(more);
      }
      return true;
    }
  }
  return false;
}

// ------------------------------------------------------------------- chunks of pairs

// The views' shares of the sorted pairs and their chunks.  A view's nearest pairs are its
// largest ones (up to all its tile rows each, where the average is three), so its first
// P.heads chunks hold only P.head_pairs pairs, and the batch takes all views' head chunks
// first (kHeadChunks of them; fewer or none where the workspace has no room for their counts).
//  The other chunks' length is the smallest power of two in [cp_lo, cp_hi] that leaves
// no more than `target` chunks: short lists still give every SM work, long ones amortise a
// chunk's scans and write longer runs.

struct ViewTab {
  uint32_t start[RAYGS_MAX_VIEWS + 1];   // first sorted pair of the view
  uint32_t chunk0[RAYGS_MAX_VIEWS + 1];  // chunks of the views before it
  uint32_t head0[RAYGS_MAX_VIEWS + 1];   // head chunks of the views before it
  uint32_t entry0[RAYGS_MAX_VIEWS + 1];  // its first count (tile rows x chunks)
  uint32_t cp, head_pairs;
  // End of the spans of unbounded supports.  With more of their rows than the capacity none of them has a span:
  // which ones found room is not the same from call to call.
  uint32_t span_end;
};

__device__ __forceinline__ void build_view_tab(const PlaceParams &P, ViewTab &T) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const uint32_t nvis = P.counters->n_visible;
    const unsigned long long span_rows = P.counters->n_span_rows;
    uint32_t cp = P.cp_lo;
    while (cp < P.cp_hi && nvis / cp >= P.target) cp <<= 1;
    uint32_t s0 = 0, c0 = 0, h0 = 0, e0 = 0;
    for (int h = 0; h < P.n_views; h += 32) {
      const int v = h + lane;
      const bool in = v < P.n_views;
      const uint32_t n = in ? (P.view_count ? P.view_count[v] : nvis) : 0u;
      const uint32_t nh = min(P.heads, (n + P.head_pairs - 1) / P.head_pairs);
      const uint32_t nch = nh + (n > nh * P.head_pairs ? (n - nh * P.head_pairs + cp - 1) / cp : 0u);
      const uint32_t e = in ? nch * uint32_t(P.cams[v].tiles_y) : 0u;
      const uint32_t si = warp_incl_scan(n), ci = warp_incl_scan(nch), hi = warp_incl_scan(nh), ei = warp_incl_scan(e);
      if (in) {
        T.start[v] = s0 + si - n;
        T.chunk0[v] = c0 + ci - nch;
        T.head0[v] = h0 + hi - nh;
        T.entry0[v] = e0 + ei - e;
      }
      s0 += __shfl_sync(0xffffffffu, si, 31);
      c0 += __shfl_sync(0xffffffffu, ci, 31);
      h0 += __shfl_sync(0xffffffffu, hi, 31);
      e0 += __shfl_sync(0xffffffffu, ei, 31);
    }
    if (lane == 0) {
      T.start[P.n_views] = s0;
      T.chunk0[P.n_views] = c0;
      T.head0[P.n_views] = h0;
      T.entry0[P.n_views] = e0;
      T.cp = cp;
      T.head_pairs = P.head_pairs;
      T.span_end = span_rows <= P.cap ? P.cap : 0u;
    }
  }
  __syncthreads();
}

struct Chunk {
  int v;               // view
  uint32_t cc, nch;    // index in the view, the view's chunks
  uint32_t q0, q1, cp; // pairs [q0, q1), at most cp
};

// Chunk c of the batch (the views' head chunks first, then their other chunks).  Whole warps.
__device__ __forceinline__ Chunk chunk_at(const ViewTab &T, int n_views, uint32_t c) {
  const int lane = threadIdx.x & 31;
  const uint32_t heads = T.head0[n_views];
  const bool head = c < heads;
  // the last view whose first chunk of this kind is not past c
  int v = -1;
  for (int h = 0; h < n_views; h += 32) {
    const int i = h + lane;
    v += __popc(__ballot_sync(0xffffffffu, i < n_views && (head ? T.head0[i] : heads + T.chunk0[i] - T.head0[i]) <= c));
  }
  Chunk k;
  k.v = v;
  const uint32_t nh = T.head0[v + 1] - T.head0[v];
  k.nch = T.chunk0[v + 1] - T.chunk0[v];
  k.cp = head ? T.head_pairs : T.cp;
  k.cc = head ? c - T.head0[v] : nh + c - (heads + T.chunk0[v] - T.head0[v]);
  k.q0 = T.start[v] + (head ? k.cc * T.head_pairs : nh * T.head_pairs + (k.cc - nh) * T.cp);
  k.q1 = min(k.q0 + k.cp, T.start[v + 1]);
  return k;
}

constexpr int kPlaceWarps = 4;  // warps per CTA, each on a chunk of its own

// tile rows of a pair, as the depth sort's last pass packs them
__device__ __forceinline__ uint32_t info_ty0(uint32_t info) { return info & 0xFFFu; }
__device__ __forceinline__ uint32_t info_rows(uint32_t info) { return ((info >> 12) & 0xFFFu) + 1u; }

// Spans of the rows of the pairs whose support is not a bounded ellipse (listed by the vertex
// stage, which also gave each its place among the spans).  One warp per pair, or up to eight
// when the pairs are few, the rows dealt out in turn: a row costs about 20 dependent segment
// tests.  Inside place_kernel such rows held up the 31 other rows of their warp and the CTA's
// barriers.
__device__ __forceinline__ void unbounded_spans(const PlaceParams &P) {
  const uint32_t n = min(P.counters->n_unbounded, P.span_list_cap);
  const int lane = threadIdx.x & 31;
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  // (from the last CTA down: the first ones count the chunks)
  const uint32_t w = (gridDim.x - 1 - blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5);
  uint32_t parts = 1;
  while (parts < 8 && uint64_t(n) * parts * 2 <= warps) parts *= 2;
  for (uint64_t u = w; u < uint64_t(n) * parts; u += warps) {
    const uint32_t pair = P.span_list[u / parts];
    if (pair == kCulled) continue;
    const Ell e = P.ell[pair];
    const uint32_t base = __float_as_uint(e.cx);
    if (base == kCulled) continue;
    const Rec &rec = P.rec[pair];
    const DevCam &cam = P.cams[pair / uint32_t(P.n)];
    const int tx0 = e.r0 & 0xFFFF, ty0 = e.r0 >> 16, tx1 = e.r1 & 0xFFFF, rows = int(e.r1 >> 16) - ty0 + 1;
    for (int r0 = 0; r0 < rows; r0 += int(parts) * 32) {
      const int r = r0 + lane * int(parts) + int(u % parts);
      const float ya = float((ty0 + r) * P.tile_h) + 0.5f;
      const float yb = float(min((ty0 + r + 1) * P.tile_h, cam.H)) - 0.5f;
      int a0 = 0, b0 = -1, state = 0;
      if (r < rows) state = support_tile_span(rec, cam, P.tile_w, ya, yb, tx0, tx1, a0, b0);
      uint32_t span = state ? uint32_t(a0) | (uint32_t(b0 - a0 + 1) << 16) : 0u;
      if (state < 0) {  // left to scan_rows; until then the span holds the pair
        span = uint32_t(tx0) | (uint32_t(tx1 - tx0 + 1) << 16);
        const uint32_t j = atomicAdd(&P.counters->n_scan, 1u);
        if (j < P.cap) {  // (always: there are no more spans)
          P.scan[j] = base + uint32_t(r);
          span = pair;
        }
      }
      if (r < rows) P.spans[base + r] = span;
    }
  }
}

// The rows that unbounded_spans left to be tested tile by tile, one warp each.
__device__ __forceinline__ void scan_rows(const PlaceParams &P) {
  const uint32_t n = min(P.counters->n_scan, P.cap);
  const uint32_t warps = gridDim.x * (blockDim.x >> 5);
  uint32_t j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  uint32_t next_slot = j < n ? P.scan[j] : 0u, next_pair = j < n ? P.spans[next_slot] : 0u;
  for (; j < n; j += warps) {
    const uint32_t slot = next_slot, pair = next_pair;
    if (j + warps < n) {  // (a span is read and then written by the one warp that tests its row)
      next_slot = P.scan[j + warps];
      next_pair = P.spans[next_slot];
    }
    const Ell e = P.ell[pair];
    const int r = int(slot - __float_as_uint(e.cx));
    const DevCam &cam = P.cams[pair / uint32_t(P.n)];
    const int ty = int(e.r0 >> 16) + r;
    int a = 0, b = -1;
    const bool any = scan_tile_span(P.rec[pair], cam, P.tile_w, float(ty * P.tile_h) + 0.5f,
                                    float(min((ty + 1) * P.tile_h, cam.H)) - 0.5f, int(e.r0 & 0xFFFF),
                                    int(e.r1 & 0xFFFF), a, b);
    if ((threadIdx.x & 31) == 0) P.spans[slot] = any ? uint32_t(a) | (uint32_t(b - a + 1) << 16) : 0u;
  }
}

// One warp per chunk (no block barriers): a difference array over the view's tile rows in
// shared memory, two atomics per pair.
template <int J>
__global__ void __launch_bounds__(32 * kPlaceWarps) pair_count_kernel(PlaceParams P, int nj_dyn) {
  await_previous();
  constexpr int NW = kPlaceWarps;
  extern __shared__ __align__(16) unsigned char s_count[];
  __shared__ ViewTab T;
  const int nj = J ? J : nj_dyn, W = 32 * nj, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t *cnt = reinterpret_cast<uint32_t *>(s_count) + warp * W;
  uint32_t *diff = reinterpret_cast<uint32_t *>(s_count) + (NW + warp) * W;
  for (int i = lane; i < W; i += 32) diff[i] = 0u;
  build_view_tab(P, T);
  const uint32_t nchunks = T.chunk0[P.n_views];
  for (uint32_t c = blockIdx.x * NW + warp; c < nchunks; c += gridDim.x * NW) {
    const Chunk k = chunk_at(T, P.n_views, c);
    const int R = P.cams[k.v].tiles_y;
    for (uint32_t q = k.q0 + lane; q < k.q1; q += 32 * 8) {
      uint32_t info[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) info[u] = q + 32 * u < k.q1 ? P.info[q + 32 * u] : kCulled;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (info[u] != kCulled) {
          atomicAdd(&diff[info_ty0(info[u])], 1u);
          atomicSub(&diff[info_ty0(info[u]) + info_rows(info[u])], 1u);
        }
    }
    __syncwarp();
    bins_counts<J>(diff, cnt, nj);
    __syncwarp();
    uint32_t *out = P.cnt1 + size_t(T.entry0[k.v]) + k.cc;
    for (int b = lane; b < R; b += 32) out[size_t(b) * k.nch] = cnt[b];
    __syncwarp();
  }
  unbounded_spans(P);
}

// One CTA per tile row: exclusive scan of its chunks' counts in place, and their total; then
// the rows left to be scanned.
__global__ void __launch_bounds__(256) row_base_kernel(PlaceParams P) {
  await_previous();
  __shared__ ViewTab T;
  __shared__ uint32_t ws[33];
  build_view_tab(P, T);
  const int t = blockIdx.x;
  int v = 0;
  while (v + 1 < P.n_views && P.cams[v + 1].trow_base <= t) ++v;
  const uint32_t nch = T.chunk0[v + 1] - T.chunk0[v];
  uint32_t *row = P.cnt1 + size_t(T.entry0[v]) + size_t(t - P.cams[v].trow_base) * nch;
  uint32_t carry = 0;
  for (uint32_t base = 0; base < nch; base += 1024) {
    uint32_t x[4], s = 0, tot;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t i = base + threadIdx.x * 4 + j;
      x[j] = i < nch ? row[i] : 0u;
      s += x[j];
    }
    uint32_t run = carry + block_excl_scan(s, ws, &tot);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t i = base + threadIdx.x * 4 + j;
      if (i < nch) row[i] = run;
      run += x[j];
    }
    carry += tot;
  }
  if (threadIdx.x == 0) P.trow_inst[t] = carry;
  scan_rows(P);
}

// Block-wide exclusive scan of 64-bit values (1024 threads).
__device__ __forceinline__ unsigned long long block_excl_scan64(unsigned long long x, unsigned long long *ws,
                                                                unsigned long long *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) ws[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const unsigned long long w = ws[lane];
    unsigned long long z = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, z, o);
      if (lane >= o) z += y;
    }
    ws[lane] = z - w;
    if (lane == 31) ws[32] = z;
  }
  __syncthreads();
  const unsigned long long r = ws[warp] + inc - x;
  *total = ws[32];
  __syncthreads();
  return r;
}

// The tile rows' ranges in the row list (one CTA; 64-bit running sums, clamped to the
// capacity: every slot below it belongs to exactly one row), the row total, the capacity
// check, the chunks of the list pass, and its instance totals cleared.
__global__ void __launch_bounds__(1024) trow_plan_kernel(PlaceParams P) {
  await_previous();
  __shared__ unsigned long long ws[33];
  const int per = (P.trows + 1023) / 1024;
  const int b = min(P.trows, int(threadIdx.x) * per), e = min(P.trows, b + per);
  unsigned long long s = 0, tot;
  for (int t = b; t < e; ++t) s += P.trow_inst[t];
  unsigned long long run = block_excl_scan64(s, ws, &tot);
  const unsigned long long cap = P.cap;
  for (int t = b; t < e; ++t) {
    const unsigned long long n = P.trow_inst[t];
    P.trow_ranges[t] = make_uint2(uint32_t(min(run, cap)), uint32_t(min(run + n, cap)));
    P.trow_inst[t] = 0ull;
    run += n;
  }
  // the chunks of the list pass: the shortest power of two in [list_lo, list_hi] that leaves
  // fewer than list_target of them (short lists still occupy every SM), at least one per tile
  // row (its tiles' ranges are written with them)
  uint32_t cr = P.list_lo;
  while (cr < P.list_hi && uint32_t(min(tot, cap)) / cr >= P.list_target) cr <<= 1;
  auto chunks = [&](int t) {
    const uint2 rr = P.trow_ranges[t];  // (this thread wrote it)
    return max(1u, (rr.y - rr.x + cr - 1) / cr);
  };
  s = 0;
  for (int t = b; t < e; ++t) s += chunks(t);
  unsigned long long nchunks;
  run = block_excl_scan64(s, ws, &nchunks);
  for (int t = b; t < e; ++t) {
    P.chunk_base[t] = uint32_t(run);
    run += chunks(t);
  }
  if (threadIdx.x == 0) {
    P.chunk_base[P.trows] = uint32_t(min(nchunks, (unsigned long long)P.max_chunks));
    P.counters->chunk_rows = cr;
  }
  if (threadIdx.x == 0) {
    P.counters->n_rows = tot;
    P.counters->n_rows_clamped = uint32_t(min(tot, cap));
    P.counters->n_rows_kept = 0u;
    P.counters->n_scan = 0u;
    P.counters->longest = 0u;
    for (int c = 0; c < kTileClasses; ++c) P.counters->tile_class[c] = 0u;
    P.counters->n_partials = 0u;
    if (tot > cap) P.counters->overflow = 1u;
  }
}

// The rows of the pairs, one warp per chunk, no barriers.  The chunk's cursor in each tile row
// starts after the rows of the chunks before; 32 pairs at a time are expanded (bins.cuh) and
// every row written to its slot (L2 merges the 8-byte stores of a chunk's run of rows in a tile
// row).  On the 3M-primitive stereo batch (17.4 M pairs, 54 M rows) 1.05 ms, 63 us on one
// headset pair of 1M primitives: bound by the gather of the support sectors in depth order
// (each 32-byte sector brings 128 bytes from DRAM, 2.4 GB in all) and the shared-memory
// latency of the expansion (43 % of issue slots).  Chunks shared by the eight warps of a CTA,
// with their rows staged in shared memory and written out in runs, took 1.15 ms and 75 us (the
// tables of 160 bins per warp cost more than the rows of a short share); chunks of 512 and 1,024
// pairs 1.30 and 1.94 ms (more views in flight than L2 holds); one 32-byte load per sector
// instead of two 16-byte ones, and 40 instead of 36 warps per SM, changed nothing.
//
// The next pairs' support sectors are loaded one group ahead, their ids two: each load is issued
// a whole group before it is needed.
//
// BWD (plans with the backward): every row also gets the position of its first instance
// among the partial sums, counted from the start of its chunk (whose base in the partials is
// allocated when the chunk is done), and every pair its run of partials.
template <int J>
static size_t place_smem(int nj) {
  const size_t W = 32 * size_t(J ? J : nj), NW = kPlaceWarps;
  return NW * (W * (J ? 12 : 8) + 32 * 48);
}

template <int J, bool BWD>
__global__ void __launch_bounds__(32 * kPlaceWarps) place_kernel(PlaceParams P, int nj_dyn) {
  await_previous();
  constexpr int NW = kPlaceWarps, U = 4;  // U: rows per lane and step of the run-time table's passes
  extern __shared__ __align__(16) unsigned char s_place[];
  __shared__ ViewTab T;
  const int nj = J ? J : nj_dyn, W = 32 * nj;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float4 *s_A = reinterpret_cast<float4 *>(s_place) + warp * 32;                      // cx, cy, a, b
  float4 *s_B = reinterpret_cast<float4 *>(s_place) + (NW + warp) * 32;               // det, hy, ydx, -
  uint4 *s_C = reinterpret_cast<uint4 *>(s_place) + (2 * NW + warp) * 32;             // start, ty0, tx0 | tx1 << 16, pos
  uint2 *mc = reinterpret_cast<uint2 *>(s_place + 48 * 32 * NW) + warp * W;           // masks and cursors
  uint32_t *tog = reinterpret_cast<uint32_t *>(s_place + 48 * 32 * NW + 8 * NW * W) + warp * W;  // toggles (J > 0)
  const int tw_shift = 31 - __clz(P.tile_w);                        // tile widths are powers of two
  const float th = float(P.tile_h);
  if (J)
    for (int i = lane; i < W; i += 32) tog[i] = 0u;
  build_view_tab(P, T);
  const uint32_t nchunks = T.chunk0[P.n_views], cap = P.cap;
  uint32_t kept = 0;
  for (uint32_t c = blockIdx.x * NW + warp; c < nchunks; c += gridDim.x * NW) {
    const Chunk ck = chunk_at(T, P.n_views, c);
    const DevCam &cam = P.cams[ck.v];
    const int R = cam.tiles_y;
    const float fH = float(cam.H);
    const uint32_t b = ck.q1;
    auto load_ids = [&](uint32_t q, uint32_t &info, uint32_t &pos, uint32_t &id) {
      info = q < b ? P.info[q] : 0u;
      id = q < b ? P.ids[q] : 0u;
      pos = q < b && P.pos ? P.pos[q] : q;
    };
    uint32_t info0, pos0, id0, info1, pos1, id1;
    Ell el;
    load_ids(ck.q0 + lane, info0, pos0, id0);
    load_ids(ck.q0 + 32 + lane, info1, pos1, id1);
    if (ck.q0 + lane < b) el = P.ell[id0];
    uint32_t cur[J ? J : 1];
    const uint32_t *cnt1 = P.cnt1 + size_t(T.entry0[ck.v]) + ck.cc;
    const uint2 *ranges = P.trow_ranges + cam.trow_base;
    auto slot = [&](int x) {  // the bin's first list slot, at most cap
      if (x >= R) return cap;
      const uint32_t st = ranges[x].x, l = cnt1[size_t(x) * ck.nch];
      return l < cap - st ? st + l : cap;
    };
    if (J) {
#pragma unroll
      for (int j = 0; j < (J ? J : 1); ++j) cur[j] = slot(lane * nj + j);
    } else {
      for (int i = lane; i < W; i += 32) mc[i] = make_uint2(0u, kCulled);  // no cursor yet
      __syncwarp();
    }
    uint32_t e_run = 0;  // BWD: instances of this chunk so far
    for (uint32_t q = ck.q0; q < b; q += 32) {
      const bool valid = q + lane < b;
      const uint32_t ty0 = info_ty0(info0), rows = valid ? info_rows(info0) : 0u;
      const uint32_t inc = warp_incl_scan(rows), start = inc - rows;
      const uint32_t n_inst = __shfl_sync(0xffffffffu, inc, 31);
      if (valid) {
        if (J) {
          atomicXor(&tog[ty0], 1u << lane);
          atomicXor(&tog[ty0 + rows], 1u << lane);
        }
        const Band bd = band_of(el);
        s_A[lane] = make_float4(bd.cx, bd.cy, bd.a, bd.b);
        s_B[lane] = make_float4(bd.det, bd.hy, bd.ydx, 0.f);
        s_C[lane] = make_uint4(start, ty0, (el.r0 & 0xFFFFu) | (el.r1 << 16), pos0);
      }
      // the groups ahead
      if (q + 32 + lane < b) el = P.ell[id1];
      info0 = info1; pos0 = pos1;
      load_ids(q + 64 + lane, info1, pos1, id1);
      __syncwarp();
      if constexpr (J > 0) {
        bins_masks<J>(tog, mc, cur);
      } else {
        // the first of the group's rows in a tile row also fetches its cursor, if the chunk had none there yet
        uint32_t seen = 0;
        for (uint32_t base = 0; base < n_inst; base += 32 * U) {
          uint32_t ty[U], at[U];
          bool fetch[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int k = instance_owner(start, valid, base + 32 * u, seen);
            const uint32_t i = base + 32 * u + lane;
            ty[u] = i < n_inst ? s_C[k].y + (i - s_C[k].x) : 0u;
            fetch[u] = i < n_inst && atomicOr(&mc[ty[u]].x, 1u << k) == 0u && mc[ty[u]].y == kCulled;
          }
#pragma unroll
          for (int u = 0; u < U; ++u) at[u] = fetch[u] ? slot(int(ty[u])) : 0u;
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (fetch[u]) mc[ty[u]].y = at[u];
        }
        __syncwarp();
      }
      uint32_t seen = 0;
      for (uint32_t base = 0; base < n_inst; base += 32) {
        int k = instance_owner(start, valid, base, seen);
        const uint32_t i = base + lane;
        if (i >= n_inst) k = 0;
        const uint4 C = s_C[k];
        const float4 A = s_A[k], B = s_B[k];
        const uint32_t ty = C.y + (i - C.x), tx0 = C.z & 0xFFFFu, tx1 = C.z >> 16;
        uint32_t len = 0, xa_t = 0;
        if (A.z > 0.f) {
          const float y0 = float(ty) * th;  // first pixel row of the tile row (exact)
          const Band bd = {A.x, A.y, A.z, A.w, B.x, B.y, B.z};
          float xa, xb;
          if (ellipse_band(bd, (y0 + 0.5f) - 0.02f, (fminf(y0 + th, fH) - 0.5f) + 0.02f, xa, xb)) {
            // pixel centres i + 0.5 in [xa, xb] (with a margin), as tile columns (the
            // conversions round up and down, and saturate)
            const int fa = __float2int_ru(xa - 0.52f), fb = __float2int_rd(xb - 0.48f);
            const uint32_t ta = max(tx0, uint32_t(max(fa, 0)) >> tw_shift);
            const uint32_t tb = min(tx1, uint32_t(max(fb, 0)) >> tw_shift);
            if (fa <= fb && fb >= 0 && ta <= tb) {
              xa_t = ta;
              len = tb - ta + 1;
            }
          }
        } else if (i < n_inst) {
          // not a bounded ellipse: the span that pair_count_kernel computed, or the whole
          // rectangle row (exact anti-aliasing bounds)
          const uint32_t sb = __float_as_uint(A.x);
          const uint32_t sp = A.z == -2.f ? tx0 | ((tx1 - tx0 + 1) << 16) : sb < T.span_end ? P.spans[sb + (i - C.x)] : 0u;
          xa_t = sp & 0xFFFFu;
          len = sp >> 16;
        }
        if (i >= n_inst) len = 0;
        kept += len ? 1u : 0u;
        uint32_t e_at = 0;
        if (BWD) {
          const uint32_t li = warp_incl_scan(len);
          e_at = e_run + li - len;
          e_run += __shfl_sync(0xffffffffu, li, 31);
          if (i < n_inst) {
            const uint32_t next = s_C[min(k + 1, 31)].x;
            const bool last_of_pair = k < 31 && q + k + 1 < b ? i + 1 == next : i + 1 == n_inst;
            uint32_t *pe = reinterpret_cast<uint32_t *>(P.pair_e + C.w);
            if (i == C.x) {
              pe[0] = e_at;
              pe[2] = c;
            }
            if (last_of_pair) pe[1] = e_at + len;
          }
        }
        if (i < n_inst) {
          const uint2 m = mc[ty];
          const uint32_t dst = m.y + __popc(m.x & ((1u << k) - 1u));
          if (dst < cap) {
            P.rows[dst] = make_uint2(C.w, xa_t | (len << 16));
            if (BWD) P.row_e[dst] = make_uint2(c, e_at);
          }
        }
      }
      __syncwarp();
      if (!J) {  // the lowest row of each mask moves the cursor past them all
        uint32_t seen = 0;
        for (uint32_t base = 0; base < n_inst; base += 32 * U) {
          uint32_t ty[U], n[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int k = instance_owner(start, valid, base + 32 * u, seen);
            const uint32_t i = base + 32 * u + lane;
            ty[u] = i < n_inst ? s_C[k].y + (i - s_C[k].x) : 0u;
            const uint32_t m = i < n_inst ? mc[ty[u]].x : 0u;
            n[u] = (m & ((1u << k) - 1u)) == 0u ? __popc(m) : 0u;
          }
          __syncwarp();
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (n[u]) mc[ty[u]] = make_uint2(0u, mc[ty[u]].y + n[u]);
          __syncwarp();
        }
      }
    }
    if (BWD && lane == 0) P.e_base[c] = atomicAdd(&P.counters->n_partials, e_run);
  }
  kept = __reduce_add_sync(0xffffffffu, kept);
  if (lane == 0 && kept) atomicAdd(&P.counters->n_rows_kept, kept);
}

// ------------------------------------------------------------------------- launchers

// Pairs of the shortest chunk: the counts (tile rows x chunks) stay within one word per (primitive, view)
// pair, and `heads` + 1 per tile row.  With more tile rows than the compiled tables hold, chunks of so many pairs
// leave most of the chip idle: where the workspace may grow, they are as short as 64 MB of counts allow, or
// 16 words per pair up to 256 MB.
uint32_t place_chunk_lo(uint64_t pairs, int max_rows, bool short_chunks) {
  uint32_t cp = 64, lo = 64;
  while (cp < uint32_t(max_rows)) cp <<= 1;
  if (!short_chunks || bins_per_lane(max_rows) <= 9) return cp;
  const uint64_t words = std::max({pairs, std::min<uint64_t>(16 * pairs, uint64_t(64) << 20), uint64_t(16) << 20});
  while (lo < cp && pairs / lo * uint64_t(max_rows) > words) lo <<= 1;
  return lo;
}
// Head chunks of a view, and one chunk that is not full.
static uint64_t place_view_chunks(int n_views, uint64_t pairs, int heads) {
  const uint64_t n = n_views > 0 ? pairs / uint64_t(n_views) : 0;
  return std::min<uint64_t>(uint64_t(heads), n / place_head_pairs(heads) + 1) + 1;
}
// Head chunks of a plan, of 2,048 pairs of a view in all: on views with more tile rows than the compiled
// tables hold its nearest pairs have up to thousands of rows each, and there are four times as many where the
// workspace may grow (64 MB of counts).
int place_heads(int max_rows, int64_t trows, bool short_chunks) {
  int heads = kHeadChunks;
  if (short_chunks && bins_per_lane(max_rows) > 9)
    while (heads < 4 * kHeadChunks && trows * heads * 2 <= int64_t(16) << 20) heads *= 2;
  return heads;
}
uint32_t place_head_pairs(int heads) { return heads > kHeadChunks ? uint32_t(16 * kHeadChunks / heads) : 16u; }
uint64_t place_max_chunks(int n_views, uint64_t pairs, uint32_t chunk_lo, int heads) {
  return pairs / chunk_lo + uint64_t(n_views) * place_view_chunks(n_views, pairs, heads);
}
uint64_t place_max_counts(int n_views, uint64_t pairs, int max_rows, int64_t trows, uint32_t chunk_lo, int heads) {
  return pairs / chunk_lo * uint64_t(max_rows) + uint64_t(trows) * place_view_chunks(n_views, pairs, heads);
}

template <int J, bool BWD>
static cudaError_t run_place(const PlaceParams &P, int nj, int num_sms, uint64_t max_chunks, cudaStream_t st) {
  constexpr int NW = kPlaceWarps;
  const size_t smem = place_smem<J>(nj), csmem = size_t(NW) * 32 * (J ? J : nj) * 8;
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024)
    e = cudaFuncSetAttribute(place_kernel<J, BWD>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e == cudaSuccess && csmem > 48 * 1024)
    e = cudaFuncSetAttribute(pair_count_kernel<J>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(csmem));
  if (e != cudaSuccess) return e;
  const uint64_t ctas = (max_chunks + NW - 1) / NW;
  launch(pair_count_kernel<J>, unsigned(std::min<uint64_t>(ctas, uint64_t(num_sms) * 8)), 32 * NW, csmem, st, P, nj);
  launch(row_base_kernel, P.trows, 256, 0, st, P);
  launch(trow_plan_kernel, 1, 1024, 0, st, P);
  launch(place_kernel<J, BWD>, unsigned(std::min<uint64_t>(ctas, uint64_t(num_sms) * 16)), 32 * NW, smem, st, P, nj);
  return cudaGetLastError();
}

cudaError_t launch_place(PlaceParams P, int num_sms, cudaStream_t st) {
  if (P.trows == 0) return cudaSuccess;
  P.cp_hi = std::max(256u, P.cp_lo);
  P.head_pairs = place_head_pairs(int(P.heads));
  P.target = uint32_t(num_sms) * 32;
  const uint64_t max_chunks =
      std::max<uint64_t>(1, place_max_chunks(P.n_views, uint64_t(P.n) * uint64_t(P.n_views), P.cp_lo, int(P.heads)));
  const int nj = bins_per_lane(P.max_rows);
  const bool bwd = P.row_e != nullptr;
#define RAYGS_PLACE(J) \
  return bwd ? run_place<J, true>(P, nj, num_sms, max_chunks, st) : run_place<J, false>(P, nj, num_sms, max_chunks, st)
  if (nj <= 1) RAYGS_PLACE(1);
  if (nj <= 3) RAYGS_PLACE(3);
  if (nj <= 5) RAYGS_PLACE(5);
  if (nj <= 9) RAYGS_PLACE(9);
  RAYGS_PLACE(0);
#undef RAYGS_PLACE
}

}  // namespace raygs
