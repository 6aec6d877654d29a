// Per-tile rasterisation with the exact, pixel-dependent anti-aliasing of Sec. 5: the
// pixel-invariant Sigma^ of Eq. mip replaced by Sigma^_x = Sigma + sigma_x^2 tau(x)^2 I and
// the modulation sqrt(|Sigma| x^T Sigma^-1 x / (|Sigma^_x| x^T Sigma^_x^-1 x)) evaluated for
// every pixel ray.  Work distribution, record pipeline, compositing and termination are
// those of the plain rasteriser (render.cu); the record is two 64-byte halves (rec, recx)
// whose fields are described with MipxOut in preprocess.cu.  Per pixel, with delta the
// offset from the projected centre:
//   y_k = b_k + g_k . delta, e_k = A_k . delta, t = m . y / |y|^2   (tau under Sigma, ray
//   x = (X, Y, 1)), l = t^2 / |x|, u_k = 1 + l w_k
//   Num = sum u_k e_k^2, Den = sum y_k^2 prod_{j != k} u_j
//   contributes iff t > 0, sum m_k y_k prod_{j != k} u_j > 0 (tau^ > 0) and
//   omega = o sqrt(|y|^2 / Den) exp(-Num / (2 Den)) >= p_min; the test Num <= kappa Den
//   (the modulation never exceeds 1) rejects first without a division.
#include "raygs_internal.cuh"
#include "raster_math.cuh"

namespace raygs {

// Tiles of TW x TH pixels in regions of RW x RH, PX pixels per thread (the region shapes and the
// claiming of items are those of render.cu).
template <int TW, int TH, int RW, int RH, int PX, bool COUNT>
__global__ void __launch_bounds__(RW *RH / PX, PX >= 4 ? 8 : PX == 2 ? 10 : 14) render_mipx_kernel(RenderParams P) {
  await_previous();
  constexpr int NT = RW * RH / PX;  // threads; one record per thread and batch
  constexpr int GX = RW / (4 * PX), PX_X = TW / RW, PARTS = PX_X * (TH / RH);
  static_assert(GX * 4 * PX == RW && RH % 8 == 0, "region shape");
  __shared__ float4 s_S[7][NT];
  __shared__ Rec s_raw[2][NT];
  __shared__ TileItems s_items;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  tile_items(P, s_items);
  for (;;) {
  if (tid == 0) claim_item<PARTS>(P, s_items);
  __syncthreads();
  const int tile = s_items.tile, part = s_items.part;
  if (tile < 0) break;
  const DevCam &cam = P.cams[s_items.view];
  const int local = tile - cam.tile_base;
  const int ty = local / cam.tiles_x, tx = local - ty * cam.tiles_x;
  const int px0 = tx * TW, py0 = ty * TH;
  const int col = (part % PX_X) * (RW / 4) + (warp % GX) * PX, row = (part / PX_X) * RH + (warp / GX) * 8;
  const int lx = lane & 3, ly = row + (lane >> 2);
  const int px = px0 + 4 * col + lx, py = py0 + ly;
  constexpr int QX = 4;  // a row's pixels lie in four interleaved columns
  const uint2 rg = P.ranges[tile];
  const float ox_tile = float(px0) + 0.5f, oy_tile = float(py0) + 0.5f;
  const float fl_x = float(lx), fl_y = float(ly), step = float(QX), skip = float(col);
  const float c2h = 0.5f * kLog2e;

  float T[PX], C0[PX], C1[PX], C2[PX], ixn[PX];
  int last[PX];
  uint32_t alive = 0;
  const float Yr = (float(py) + 0.5f - cam.cy) * cam.ify;
#pragma unroll
  for (int k = 0; k < PX; ++k) {
    T[k] = 1.f; C0[k] = 0.f; C1[k] = 0.f; C2[k] = 0.f; last[k] = 0;
    if (py < cam.H && px + k * QX < cam.W) alive |= 1u << k;
    const float Xr = (float(px + k * QX) + 0.5f - cam.cx) * cam.ifx;
    ixn[k] = rsqrtf(fmaf(Xr, Xr, fmaf(Yr, Yr, 1.f)));  // 1 / |x|
  }
  const uint32_t inside = alive;
  unsigned long long n_eval = 0, n_comp = 0;

  // two-stage pipeline as in render.cu: raw halves of the next batch in flight (cp.async),
  // pair indices of the batch after that in a register
  uint32_t nxt;
  {
    const uint32_t i = rg.x + tid;
    if (i < rg.y) {
      const uint32_t pr = P.pairs[P.inst_vals[i]];
      cp_async_rec(&s_raw[0][tid], &P.rec[pr]);
      cp_async_rec(&s_raw[1][tid], &P.recx[pr]);
    }
    cp_async_commit();
    const uint32_t i2 = rg.x + NT + tid;
    nxt = i2 < rg.y ? P.pairs[P.inst_vals[i2]] : 0u;
  }

  for (uint32_t start = rg.x; start < rg.y; start += NT) {
    if (__syncthreads_and(alive == 0)) break;
    cp_async_wait_all();
    if (start + tid < rg.y) {
      const Rec &r = s_raw[0][tid], &q = s_raw[1][tid];
      const df ox = two_sum(ox_tile, -r.a.x);
      const df oy = two_sum(oy_tile, -r.a.y);
      s_S[0][tid] = make_float4(__fadd_rn(ox.hi, __fsub_rn(ox.lo, r.a.z)),
                                __fadd_rn(oy.hi, __fsub_rn(oy.lo, r.a.w)), r.b.x, r.b.y);
      s_S[1][tid] = make_float4(r.b.z, r.b.w, r.c.x, r.c.y);
      s_S[2][tid] = make_float4(r.c.z, r.c.w, r.d.x, r.d.y);
      s_S[3][tid] = make_float4(r.d.z, r.d.w, q.a.x, q.a.y);
      s_S[4][tid] = make_float4(q.a.z, q.b.x, q.b.y, q.b.z);
      s_S[5][tid] = make_float4(q.c.x, q.c.y, q.c.z, q.a.w);
      s_S[6][tid] = make_float4(q.b.w, q.d.x, q.d.y, q.d.z);
    }
    __syncthreads();
    {
      const uint32_t i = start + NT + tid;
      if (i < rg.y) {
        cp_async_rec(&s_raw[0][tid], &P.rec[nxt]);
        cp_async_rec(&s_raw[1][tid], &P.recx[nxt]);
      }
      cp_async_commit();
      const uint32_t i2 = start + 2 * NT + tid;
      nxt = i2 < rg.y ? P.pairs[P.inst_vals[i2]] : 0u;
    }
    const int nb = min(NT, int(rg.y - start));
    for (int j = 0; j < nb && alive; ++j) {
      const float4 S0 = s_S[0][j], S1 = s_S[1][j], S2 = s_S[2][j], S3 = s_S[3][j];
      const float4 S4 = s_S[4][j], S5 = s_S[5][j];
      if (COUNT) n_eval += __popc(alive);
      const float dy = S0.y + fl_y;
      const float dx0 = S0.x + fl_x;
      // row terms of the affine forms
      const float e0r = S0.w * dy, e1r = S1.y * dy, e2r = S1.w * dy;
      const float y0r = fmaf(S2.y, dy, S3.z), y1r = fmaf(S2.w, dy, S3.w), y2r = fmaf(S3.y, dy, S4.x);
      float om[PX];
      uint32_t hit = 0;
#pragma unroll
      for (int k = 0; k < PX; ++k) {
        const float dx = dx0 + (skip + float(k)) * step;
        const float e0 = fmaf(S0.z, dx, e0r), e1 = fmaf(S1.x, dx, e1r), e2 = fmaf(S1.z, dx, e2r);
        const float y0 = fmaf(S2.x, dx, y0r), y1 = fmaf(S2.z, dx, y1r), y2 = fmaf(S3.x, dx, y2r);
        const float my0 = S4.y * y0, my1 = S4.z * y1, my2 = S4.w * y2;
        const float tn = my0 + my1 + my2;
        const float yy = fmaf(y0, y0, fmaf(y1, y1, y2 * y2));
        const float t = __fdividef(tn, yy);
        const float l = t * t * ixn[k];
        const float u0 = fmaf(l, S5.x, 1.f), u1 = fmaf(l, S5.y, 1.f), u2 = fmaf(l, S5.z, 1.f);
        const float u12 = u1 * u2, u02 = u0 * u2, u01 = u0 * u1;
        const float num = fmaf(u0 * e0, e0, fmaf(u1 * e1, e1, u2 * e2 * e2));
        const float den = fmaf(y0 * y0, u12, fmaf(y1 * y1, u02, y2 * y2 * u01));
        const float sg = fmaf(my0, u12, fmaf(my1, u02, my2 * u01));
        om[k] = 0.f;
        if (tn > 0.f && sg > 0.f && num <= s_S[6][j].x * den) {
          const float iden = __fdividef(1.f, den);
          const float lg = __log2f(yy * iden);
          const float w = ex2_approx(fmaf(0.5f, lg, S5.w) - c2h * num * iden);
          om[k] = w;
          if (w >= P.p_min) hit |= 1u << k;
        }
      }
      hit &= alive;
      if (hit) {
        const float4 S6 = s_S[6][j];
#pragma unroll
        for (int k = 0; k < PX; ++k) {
          if (hit & (1u << k)) {
            const float al = fminf(P.alpha_max, om[k]);
            const float w = al * T[k];
            const float Tn = T[k] - w;
            if (Tn < P.t_stop) {
              alive &= ~(1u << k);
            } else {
              C0[k] = fmaf(w, S6.y, C0[k]);
              C1[k] = fmaf(w, S6.z, C1[k]);
              C2[k] = fmaf(w, S6.w, C2[k]);
              T[k] = Tn;
              last[k] = int(start - rg.x) + j + 1;
              if (COUNT) ++n_comp;
            }
          }
        }
      }
    }
  }
  cp_async_wait_all();  // no copy may outlive the block
  if (inside) {
    const long long pix = cam.pix_base + (long long)py * cam.W + px;
#pragma unroll
    for (int k = 0; k < PX; ++k) {
      if (inside & (1u << k)) {
        const long long o = pix + k * QX;
        P.rgb[3 * o] = C0[k];
        P.rgb[3 * o + 1] = C1[k];
        P.rgb[3 * o + 2] = C2[k];
        if (P.Tf) P.Tf[o] = T[k];
        if (P.ncontrib) P.ncontrib[o] = last[k];
      }
    }
  }
  if (COUNT) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n_eval += __shfl_down_sync(0xffffffffu, n_eval, o);
      n_comp += __shfl_down_sync(0xffffffffu, n_comp, o);
    }
    if ((tid & 31) == 0) {
      atomicAdd(&P.eval_counts[0], n_eval);
      atomicAdd(&P.eval_counts[1], n_comp);
    }
  }
  __syncthreads();  // shared state is free before the next claim
  }
  leave_items(P);
}

// Two pixels per thread: at four the kernel needs 117 registers (8 CTAs of 64 threads per SM) and
// was the slower one at every size (500k primitives: 458 against 350-373 us at 1280x720, 609
// against 521 at 1920x1080, 901 against 776 at 2560x1440; 1M at 3840x2160 2.28 against 1.96 ms).
// By the tiles (of 16x16 pixels) per slot of 16 CTAs per SM, as in render.cu: up to 0.75, 8x8 blocks with
// one pixel per thread (640x360, 200k primitives, 0.4: 285 us, two pixels 358 to 428; 160x120, 20k: 121
// against 172), where the longest list sets the time; up to 2.5, 8x8 blocks with two (720p, 1.5: 350
// against 373 in 8x16; with 1.5M primitives 504 against 517); else 8x16 regions (1080p, 3.4: 521
// against 529; 4K, 13: 1.96 against 2.02 ms).  Measured on 16x16 tiles; the regions are the same in every
// tile shape (a 640x360 view with 100k primitives 156 us, with 16x8 tiles 129, 32x16 210, 8x8 95).
template <int TW, int TH, int PX>
static cudaError_t run_mipx(const RenderParams &P, int num_sms, bool count, cudaStream_t st) {
  constexpr int RW = TH >= 16 ? 8 : TW >= 16 ? 16 : 8, RH = TH >= 16 ? 16 : 8;
  constexpr int BLOCKS = (TW / 8) * (TH / 8);
  const int64_t area = int64_t(P.n_tiles) * TW * TH, slots = int64_t(num_sms) * 16 * 256;
  if (count) launch_persistent(render_mipx_kernel<TW, TH, TW, TH, PX, true>, TW * TH / PX, 1, num_sms, P, st);
  else if (4 * area <= 3 * slots) launch_persistent(render_mipx_kernel<TW, TH, 8, 8, 1, false>, 64, BLOCKS, num_sms, P, st);
  else if (2 * area <= 5 * slots) launch_persistent(render_mipx_kernel<TW, TH, 8, 8, 2, false>, 32, BLOCKS, num_sms, P, st);
  else launch_persistent(render_mipx_kernel<TW, TH, RW, RH, 2, false>, RW * RH / 2, BLOCKS * 64 / (RW * RH), num_sms, P, st);
  return cudaGetLastError();
}

cudaError_t launch_render_mipx(const RenderParams &P, int tile_w, int tile_h, int num_sms, bool count,
                               cudaStream_t st) {
  if (P.n_tiles <= 0) return cudaSuccess;
  if (tile_w == 16 && tile_h == 16) return run_mipx<16, 16, 4>(P, num_sms, count, st);
  if (tile_w == 16 && tile_h == 8) return run_mipx<16, 8, 4>(P, num_sms, count, st);
  if (tile_w == 32 && tile_h == 16) return run_mipx<32, 16, 8>(P, num_sms, count, st);
  if (tile_w == 8 && tile_h == 8) return run_mipx<8, 8, 2>(P, num_sms, count, st);
  return cudaErrorInvalidValue;
}

}  // namespace raygs
