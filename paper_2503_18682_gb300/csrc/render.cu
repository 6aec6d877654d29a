// Per-tile rasterisation and front-to-back compositing (Sec. 3 Eq. rendering and
// Eq. rend_opacity; Sec. 4.2 fragment formula).
//
// Persistent CTAs (one per resident slot) take the screen tiles of all views one at a time,
// those with the longest lists first; each thread shades PX pixels of a tile row.  A tile's
// instance list (depth order) is consumed in batches: each thread stages records in shared memory, converting the projected centre to a tile-relative
// offset in double-float so that per-pixel offsets stay exact to the float32 rounding of
// the offset itself.  Per pixel, with delta = pixel centre - projected centre:
//   y01 = G delta, y2 = 1 + h . delta, q = |y01|^2, r = y2^2
//   contributes iff y2 > 0 and kp q - r <= 0          (D <= kappa, Eq. support)
//   D log2(e)/2 = c2h q / (q + r)                     (fragment formula)
//   omega = min(alpha_max, 2^(log2 o - D log2(e)/2))
// With the GS divergence of Sec. 3.1 the records carry h = 0 and G with G^T G = Sigma_pi^-1,
// so that r = 1, the test reads q <= kappa and D log2(e)/2 = c2h q (DIV = 1 below).  The
// records' G carries sqrt(kp), so that the support test is the single compare q' <= r.
// A thread's PX pixels lie on one tile row, interleaved with the other threads of that
// row (columns lx, lx + QX, lx + 2 QX, ...), so that a footprint covering a range of
// columns hits the same pixel slots k in every lane of the row and the per-slot
// compositing stays convergent.  The PX pixels share the row term of y and step the
// column term by QX pixels (y += QX G[:,0]).  Compositing of a pixel stops before a primitive that would take T
// below t_stop; a thread skips records once its pixels have all stopped, and the CTA
// leaves the list once every thread has.
#include "raygs_internal.cuh"
#include "raster_math.cuh"

namespace raygs {

// Compositing state of a thread's pixels.
template <int PX>
struct Pixels {
  float T[PX], C0[PX], C1[PX], C2[PX];
  int last[PX];
  uint32_t alive;
  unsigned long long n_eval, n_comp, n_iter;  // instrumented variant
};

// The batch's records (CULL: those of the warp's list), n of them, front to back.  PRE:
// interleaved columns of the row before the thread's own (compile-time: stepping over them costs
// its additions alone).
template <int PX, int PRE, bool CULL, bool COUNT, int DIV>
__device__ __forceinline__ void composite_batch(const RenderParams &P, Pixels<PX> &S, const float4 *s_A,
                                                const float4 *s_B, const float4 *s_C, const float4 *s_D,
                                                const uint8_t *list, int n, int first, float fl_x, float fl_y) {
  // two records per iteration give the scheduler independent work (8 pixels per thread
  // would spill)
#pragma unroll(PX >= 8 ? 1 : 2)
  for (int i = 0; i < n && S.alive; ++i) {
    const int j = CULL ? list[i] : i;
    const float4 A = s_A[j], B = s_B[j];
    const float4 Cc = s_C[j];
    if (COUNT) { S.n_eval += __popc(S.alive); ++S.n_iter; }
    // with 8 pixels per thread a conservative segment test pays for itself (fewer
    // pixels per thread are cheaper to test directly); the instrumented variant tests
    // every pixel, so its image checks the filters
    if (PX >= 8 && !COUNT && !row_may_hit<PX>(A, B, Cc, s_D[j].w, fl_x, fl_y, 4.f)) continue;
    float q[PX], r[PX], y0[PX], y1[PX], y2[PX];
    uint32_t hit = eval_pixels<PX, PRE>(A, B, fl_x, fl_y, 4.f, q, r, y0, y1, y2);
    hit &= S.alive;
    if (hit) {
      const float4 Dd = s_D[j];
#pragma unroll
      for (int k = 0; k < PX; ++k) {
        if (hit & (1u << k)) {
          const float al = fminf(P.alpha_max, pixel_opacity<DIV>(Cc, q[k], r[k]));
          const float w = al * S.T[k];
          const float Tn = S.T[k] - w;
          if (Tn < P.t_stop) {
            S.alive &= ~(1u << k);
          } else {
            S.C0[k] = fmaf(w, Dd.x, S.C0[k]);
            S.C1[k] = fmaf(w, Dd.y, S.C1[k]);
            S.C2[k] = fmaf(w, Dd.z, S.C2[k]);
            S.T[k] = Tn;
            S.last[k] = first + j + 1;
            if (COUNT) ++S.n_comp;
          }
        }
      }
    }
  }
}

template <int NB, int NW>
struct RasterSmem {
  float4 A[NB], B[NB], C[NB], D[NB];
  Rec raw[NB];
  uint8_t list[NW][NB];  // per warp, the batch's records it keeps 
  TileItems items;
};

// Tiles of TW x TH pixels in regions of RW x RH, PX pixels per thread; a warp shades 4 PX columns
// of eight rows.  CULL: a warp composites only the records whose support can meet one of its
// pixel centres, listed once per batch.
template <int TW, int TH, int RW, int RH, int PX, int NBF, bool CULL, bool COUNT, int DIV, typename Smem>
__device__ __forceinline__ void render_regions(const RenderParams &P, Smem &M) {
  constexpr int NT = RW * RH / PX;    // threads
  constexpr int NB = NBF * NT;        // records per batch
  constexpr int GX = RW / (4 * PX);   // warps side by side
  constexpr int PX_X = TW / RW, PARTS = PX_X * (TH / RH);
  static_assert(GX * 4 * PX == RW && RH % 8 == 0 && NB <= 256, "region shape");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float4 *s_A = M.A, *s_B = M.B, *s_C = M.C, *s_D = M.D;
  // persistent CTAs: each claims the next item until none is left
  for (;;) {
  if (tid == 0) claim_item<PARTS>(P, M.items);
  __syncthreads();
  const int tile = M.items.tile, part = M.items.part;
  if (tile < 0) break;
  const DevCam &cam = P.cams[M.items.view];
  const int local = tile - cam.tile_base;
  const int ty = local / cam.tiles_x, tx = local - ty * cam.tiles_x;
  const int px0 = tx * TW, py0 = ty * TH;
  // the warp's first column (in units of four pixels) and row in the tile
  const int col = (part % PX_X) * (RW / 4) + (warp % GX) * PX, row = (part / PX_X) * RH + (warp / GX) * 8;
  const int lx = lane & 3, ly = row + (lane >> 2);
  const int px = px0 + 4 * col + lx, py = py0 + ly;
  const uint2 rg = P.ranges[tile];
  const float ox_tile = float(px0) + 0.5f, oy_tile = float(py0) + 0.5f;
  const float fl_x = float(lx), fl_y = float(ly);

  Pixels<PX> S;
  S.alive = 0;
#pragma unroll
  for (int k = 0; k < PX; ++k) {
    S.T[k] = 1.f; S.C0[k] = 0.f; S.C1[k] = 0.f; S.C2[k] = 0.f; S.last[k] = 0;
    if (py < cam.H && px + 4 * k < cam.W) S.alive |= 1u << k;
  }
  const uint32_t inside = S.alive;
  S.n_eval = S.n_comp = S.n_iter = 0;
  uint32_t stop_at = rg.y;  // first list entry the CTA did not stage

  // Records move through a two-stage pipeline: while a batch is composited, the raw
  // records of the next batch are in flight to shared memory (cp.async) and the record
  // indices of the batch after that are being loaded into registers.
  uint32_t nxt[NBF];
#pragma unroll
  for (int rr = 0; rr < NBF; ++rr) {
    const uint32_t i = rg.x + tid + rr * NT;
    if (i < rg.y) cp_async_rec(&M.raw[tid + rr * NT], &P.rec[P.pairs[P.inst_vals[i]]]);
  }
  cp_async_commit();
#pragma unroll
  for (int rr = 0; rr < NBF; ++rr) {
    const uint32_t i = rg.x + NB + tid + rr * NT;
    nxt[rr] = i < rg.y ? P.pairs[P.inst_vals[i]] : 0u;
  }

  for (uint32_t start = rg.x; start < rg.y; start += NB) {
    if (__syncthreads_and(S.alive == 0)) {
      stop_at = start;
      break;
    }
    cp_async_wait_all();  // this thread's raw slots of the batch have landed
#pragma unroll
    for (int rr = 0; rr < NBF; ++rr) {
      const int slot = tid + rr * NT;
      if (start + slot < rg.y)
        stage_record<DIV>(M.raw[slot], ox_tile, oy_tile, M.A[slot], M.B[slot], M.C[slot], M.D[slot]);
    }
    __syncthreads();
#pragma unroll
    for (int rr = 0; rr < NBF; ++rr) {
      const uint32_t i = start + NB + tid + rr * NT;
      if (i < rg.y) cp_async_rec(&M.raw[tid + rr * NT], &P.rec[nxt[rr]]);
    }
    cp_async_commit();
#pragma unroll
    for (int rr = 0; rr < NBF; ++rr) {
      const uint32_t i = start + 2 * NB + tid + rr * NT;
      nxt[rr] = i < rg.y ? P.pairs[P.inst_vals[i]] : 0u;
    }
    const int nb = min(NB, int(rg.y - start)), first = int(start - rg.x);
    int n = nb;
    uint8_t *list = M.list[CULL ? warp : 0];
    if (CULL) {
      n = 0;
      if (__any_sync(0xffffffffu, S.alive)) {
#pragma unroll
        for (int r0 = 0; r0 < NB; r0 += 32) {
          const int r = r0 + lane;
          const bool keep = r < nb && box_may_hit(s_A[r], s_B[r], float(4 * col) + (2 * PX - 0.5f),
                                                  float(row) + 3.5f, 2 * PX - 0.5f, 3.5f);
          const uint32_t ball = __ballot_sync(0xffffffffu, keep);
          if (keep) list[n + __popc(ball & ((1u << lane) - 1u))] = uint8_t(r);
          n += __popc(ball);
        }
        __syncwarp();
      }
    }
#define RAYGS_COL(c)                                                                                           \
  case c:                                                                                                      \
    if constexpr (c < TW / (4 * PX))                                                                           \
      composite_batch<PX, (c) * PX, CULL, COUNT, DIV>(P, S, s_A, s_B, s_C, s_D, list, n, first, fl_x, fl_y);         \
    break;
    switch (TW == 4 * PX ? 0 : col / PX) {  // (the same for the whole warp)
      RAYGS_COL(0) RAYGS_COL(1) RAYGS_COL(2) RAYGS_COL(3)
      RAYGS_COL(4) RAYGS_COL(5) RAYGS_COL(6) RAYGS_COL(7)
    }
#undef RAYGS_COL
  }
  cp_async_wait_all();  // no copy may outlive the block
  const bool alive_any = COUNT ? __syncthreads_or(S.alive != 0) : false;
  if (inside) {
    const long long pix = cam.pix_base + (long long)py * cam.W + px;
#pragma unroll
    for (int k = 0; k < PX; ++k) {
      if (inside & (1u << k)) {
        const long long o = pix + 4 * k;
        P.rgb[3 * o] = S.C0[k];
        P.rgb[3 * o + 1] = S.C1[k];
        P.rgb[3 * o + 2] = S.C2[k];
        if (P.Tf) P.Tf[o] = S.T[k];
        if (P.ncontrib) P.ncontrib[o] = S.last[k];
      }
    }
  }
  if (COUNT) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      S.n_eval += __shfl_down_sync(0xffffffffu, S.n_eval, o);
      S.n_comp += __shfl_down_sync(0xffffffffu, S.n_comp, o);
      S.n_iter += __shfl_down_sync(0xffffffffu, S.n_iter, o);
    }
    if (lane == 0) {
      atomicAdd(&P.eval_counts[0], S.n_eval);
      atomicAdd(&P.eval_counts[1], S.n_comp);
      atomicAdd(&P.eval_counts[3], S.n_iter);
    }
    if (tid == 0) {
      atomicAdd(&P.eval_counts[2], (unsigned long long)(stop_at - rg.x));
      if (P.tile_stop) P.tile_stop[tile] = alive_any ? kCulled : stop_at - rg.x;
    }
  }
  __syncthreads();  // shared state is free before the next claim
  }
}

// Whole tiles, every record of the list tested by every warp: the variant for many tiles.  Listing
// each warp's records (CULL) as well made it slower on the stereo batch (4.33 against 4.05 ms):
// most of a tile's records meet both of its warps.
template <int TW, int TH, int PX, int NBF, bool COUNT, int DIV>
__global__ void __launch_bounds__(TW *TH / PX, 16) render_kernel(RenderParams P) {
  await_previous();
  __shared__ RasterSmem<NBF * TW * TH / PX, 1> M;
  tile_items(P, M.items);
  render_regions<TW, TH, TW, TH, PX, NBF, false, COUNT, DIV>(P, M);
  leave_items(P);
}

// Parts of tiles, for batches of few tiles (launch_render): there the time is that of the tiles
// with the longest lists, whose records (400 cycles each at four pixels per thread alone, 1,100
// with the SM full) are composited one after the other.  Two pixels per thread and warps of 8x8
// pixels that list their records per batch; or, when no more than a fraction of the tiles holds
// records worth speaking of, one pixel per thread in 8x8 blocks.  A pixel's arithmetic is that of
// the whole-tile kernel, bit for bit.  720p, 500k primitives: 131 us against 179 in whole tiles
// (151 with one pixel per thread), 1.5M: 174 against 217 (212); four uneven 640x480 views of 200k:
// 77 us with one pixel per thread, 117 with two, 191 in whole tiles; 64x64, 1k: 19, 29 and 48.
// Where the lists are even enough that the longest one does not set the time (large primitives, a camera
// inside them, an empty view), the most pixels per thread and no lists of the warps: 100k large
// primitives at 1280x720 117 us against 133 in parts, 5k around the camera 56 against 77, an empty
// 1600x900 view 17 against 25 (16x8 tiles 117 against 137, 60 against 76; 32x16 tiles, then in halves, 126
// against 141, 61 against 83).  The line at 0.4 of the longest list per slot: 100k middling primitives at
// 960x540 (0.34) 79 us in parts against 77, at 1280x720 (0.6) 116 against 111.
template <int TW, int TH, int NBF, int DIV>
__global__ void __launch_bounds__(64, 18) render_parts_kernel(RenderParams P) {
  await_previous();
  __shared__ RasterSmem<NBF * 64, 2> M;
  constexpr int RW = TH >= 16 ? 8 : TW >= 16 ? 16 : 8, RH = TH >= 16 ? 16 : 8, PX = RW * RH / 64;
  tile_items(P, M.items);
  // tiles with 64 records and more (class 9 is the last of them)
  static_assert(tile_class_min(9) == 64, "classes");
  const bool fine = P.class_tiles && M.items.first[10] * uint32_t((TW / 8) * (TH / 8)) <= uint32_t(P.slots);
  // the lists' sum per slot at least 0.4 of the longest one, in lists of 16x16 tiles
  const uint2 lists = M.items.lists;
  const bool even = P.class_tiles && 10ull * TW * TH * lists.x >= 4ull * 256 * uint32_t(P.slots) * lists.y;
  if (TW >= 16 && even) render_regions<TW, TH, 16, TH, TH / 4, NBF, false, false, DIV>(P, M);
  else if (PX == 1 || fine) render_regions<TW, TH, 8, 8, 1, NBF, true, false, DIV>(P, M);
  else render_regions<TW, TH, RW, RH, PX, NBF, true, false, DIV>(P, M);
  leave_items(P);
}

template <int TW, int TH, int PX, int NBF, int DIV>
static cudaError_t run_render(const RenderParams &P, int num_sms, bool count, bool parts, cudaStream_t st) {
  constexpr int NT = TW * TH / PX;
  if (count) launch_persistent(render_kernel<TW, TH, PX, NBF, true, DIV>, NT, 1, num_sms, P, st);
  else if (parts) launch_persistent(render_parts_kernel<TW, TH, NBF, DIV>, 64, (TW / 8) * (TH / 8), num_sms, P, st);
  else launch_persistent(render_kernel<TW, TH, PX, NBF, false, DIV>, NT, 1, num_sms, P, st);
  return cudaGetLastError();
}

cudaError_t launch_render(const RenderParams &P, int tile_w, int tile_h, int batch_records, int num_sms,
                          bool count, cudaStream_t st) {
  if (P.n_tiles <= 0) return cudaSuccess;
  const bool gs = P.qmix == 0.f;  // D_gs records (Sec. 3.1)
  // Parts of tiles up to 2.5 tiles of 16x16 pixels per slot of the whole-tile kernel (16 CTAs per
  // SM).  500k primitives at 1280x720 (1.5 tiles per slot) 130 against 174 us whole, 1440x810 (1.9)
  // 141 against 168, 1600x900 (2.3) 154 against 171 (2M primitives: 211 against 210); 1920x1080
  // (3.4) 194 against 187, 2560x1440 (5.9) 292 against 259.
  // On 8x8 tiles, whose parts are the tiles themselves with one instead of two pixels per thread, up to
  // 0.75: 500k primitives at 800x450 (0.59) 83 against 95 us whole, 880x495 (0.70) 91 against 94, 960x540
  // (0.84) 99 against 95, 1280x720 137 against 115, 1600x900 188 against 149.  (16x8 and 32x16 tiles at
  // 1440x810: 150 against 142, 169 against 339.)
  const int64_t area = int64_t(P.n_tiles) * tile_w * tile_h, slots = int64_t(num_sms) * 16 * 256;
  const bool parts = tile_w * tile_h <= 64 ? 4 * area <= 3 * slots : 2 * area <= 5 * slots;
#define RAYGS_RENDER_CASE(TW, TH, PX, NBF)                                                       \
  if (tile_w == TW && tile_h == TH && batch_records == NBF)                                     \
    return gs ? run_render<TW, TH, PX, NBF, 1>(P, num_sms, count, parts, st)                    \
              : run_render<TW, TH, PX, NBF, 0>(P, num_sms, count, parts, st);
  RAYGS_RENDER_CASE(16, 16, 4, 1)
  RAYGS_RENDER_CASE(16, 8, 4, 1)
  RAYGS_RENDER_CASE(32, 16, 8, 1)
  RAYGS_RENDER_CASE(8, 8, 2, 1)
  RAYGS_RENDER_CASE(16, 16, 4, 2)
  RAYGS_RENDER_CASE(16, 8, 4, 2)
  RAYGS_RENDER_CASE(32, 16, 8, 2)
  RAYGS_RENDER_CASE(8, 8, 2, 2)
#undef RAYGS_RENDER_CASE
  return cudaErrorInvalidValue;
}

}  // namespace raygs
