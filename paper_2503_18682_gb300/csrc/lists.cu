// Per-tile instance lists from the support rows listed by tile row (rows.cu).
//
// Each tile row's rows are cut into chunks, one CTA each:
//   list_count_kernel  per chunk and tile column, the chunk's instances; the last CTA to finish
//                      scans the tile rows' instance totals
//   list_kernel        the instances themselves, in depth order, and the tiles' ranges
#include <algorithm>

#include "bins.cuh"

namespace raygs {

__device__ __forceinline__ int view_of_trow(const DevCam *cams, int n_views, int t) {
  int v = 0;
  while (v + 1 < n_views && cams[v + 1].trow_base <= t) ++v;
  return v;
}

// The chunk of rows a CTA owns: tile row t (the last one whose first chunk is not past it) and
// its rows [first, last).
__device__ __forceinline__ bool chunk_of(const ListParams &P, uint32_t chunk, int &t, int &c, uint2 &rows) {
  if (chunk >= P.chunk_base[P.trows]) return false;
  int lo = 0, hi = P.trows - 1;
  while (lo < hi) {
    const int m = (lo + hi + 1) >> 1;
    if (P.chunk_base[m] <= chunk) lo = m; else hi = m - 1;
  }
  t = lo;
  c = int(chunk - P.chunk_base[t]);
  const uint32_t cr = P.counters->chunk_rows;
  const uint2 rr = P.trow_ranges[t];
  const uint32_t first = uint32_t(min((unsigned long long)rr.x + (unsigned long long)c * cr, (unsigned long long)rr.y));
  rows = make_uint2(first, first + min(cr, rr.y - first));
  return true;
}

// A row's columns, kept inside the tile row whatever the list holds.
__device__ __forceinline__ uint2 row_cols(uint32_t span, uint32_t tx) {
  const uint32_t a = min(span & 0xFFFFu, tx);
  return make_uint2(a, min(span >> 16, tx - a));
}

// Exclusive scan of the tile rows' instance totals in place by one CTA: each tile row's first
// instance, the instance total, its capacity clamp and the overflow flag.
__device__ void scan_trow_instances(const ListParams &P) {
  __shared__ unsigned long long ws[8];
  const int NT = blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long carry = 0;
  for (int base = 0; base < P.trows; base += NT * 4) {
    unsigned long long x[4], s = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = base + int(threadIdx.x) * 4 + j;
      x[j] = i < P.trows ? __ldcg(P.trow_inst + i) : 0ull;
      s += x[j];
    }
    unsigned long long inc = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) ws[warp] = inc;
    __syncthreads();
    unsigned long long run = carry + inc - s, tot = 0;
    for (int w = 0; w < NT / 32; ++w) {
      run += w < warp ? ws[w] : 0ull;
      tot += ws[w];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int i = base + int(threadIdx.x) * 4 + j;
      if (i < P.trows) P.trow_inst[i] = run;
      run += x[j];
    }
    carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    P.counters->n_instances = carry;
    P.counters->n_inst_clamped = carry > P.cap ? P.cap : uint32_t(carry);
    if (carry > P.cap) P.counters->overflow = 1u;
  }
}

// Instances per tile column of one chunk: each row covers the tile columns
// [txa, txa + len); a difference array over the columns and its prefix sum count them.
__global__ void __launch_bounds__(256) list_count_kernel(ListParams P) {
  await_previous();
  extern __shared__ uint32_t s_diff[];  // [max_tiles_x + 1]
  __shared__ uint32_t s_ws[33];
  __shared__ bool s_last;
  for (uint32_t chunk = blockIdx.x;; chunk += gridDim.x) {
    int t, c;
    uint2 rows;
    if (!chunk_of(P, chunk, t, c, rows)) break;
    const int TX = P.cams[view_of_trow(P.cams, P.n_views, t)].tiles_x;
    for (int x = threadIdx.x; x <= TX; x += blockDim.x) s_diff[x] = 0u;
    __syncthreads();
    // four rows per thread at a time, their loads issued before any of their atomics
    for (uint32_t i0 = rows.x + threadIdx.x; i0 < rows.y; i0 += 4 * blockDim.x) {
      uint32_t span[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t i = i0 + k * blockDim.x;
        span[k] = i < rows.y ? P.rows[i].y : 0u;  // 0: no tiles
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint2 cl = row_cols(span[k], uint32_t(TX));
        if (cl.y) {
          atomicAdd(&s_diff[cl.x], 1u);
          atomicSub(&s_diff[cl.x + cl.y], 1u);
        }
      }
    }
    __syncthreads();
    const int per = (TX + int(blockDim.x) - 1) / int(blockDim.x);
    const int x0 = min(TX, int(threadIdx.x) * per), x1 = min(TX, x0 + per);
    uint32_t dsum = 0;
    for (int x = x0; x < x1; ++x) dsum += s_diff[x];
    uint32_t dtot;
    uint32_t run = block_excl_scan(dsum, s_ws, &dtot);
    uint32_t *out = P.cnt2 + size_t(chunk) * size_t(P.max_tiles_x);
    unsigned long long mine = 0;
    for (int x = x0; x < x1; ++x) {
      run += s_diff[x];
      out[x] = run;
      mine += run;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&P.trow_inst[t], mine);
    __syncthreads();
  }
  // the last CTA to finish scans the totals (nothing waits: every other CTA leaves at once)
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&P.counters->lists_done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (s_last) {
    __threadfence();
    scan_trow_instances(P);
    if (threadIdx.x == 0) P.counters->lists_done = 0u;
  }
}

// Instance lists of one chunk of a tile row.  Its cursor in tile column x starts after the
// tile row's earlier tiles (all chunks) and after the earlier chunks' instances in x; chunk 0
// also writes the tile row's ranges.  Rows are then taken in sorted (depth) order, NT * KR
// at a time, in 32-row groups (KR * NT / 32 groups: row q of the step is lane q % 32 of group
// q / 32); every lane marks the tiles of its row in its group's bit mask per tile, and the
// rank of (row, tile) is the tile's running cursor plus the rows of lower groups and lower
// lanes that cover the same tile.  Each tile's list keeps depth order.  The masks are
// double-buffered (the buffer of the next step is cleared while this one is read) and the
// rows of the next step are loaded during this one.
template <int NT, int KR>
__global__ void __launch_bounds__(NT) list_kernel(ListParams P) {
  await_previous();
  constexpr int VW = NT / 32 * KR;  // row groups per step
  extern __shared__ uint32_t s_mem[];
  int grow, chunk_c;
  uint2 rr;
  if (!chunk_of(P, blockIdx.x, grow, chunk_c, rr)) return;
  const int v = view_of_trow(P.cams, P.n_views, grow);
  const DevCam &cam = P.cams[v];
  const int TX = cam.tiles_x;
  const int TP = TX | 1;                     // odd row stride: no bank conflicts down a column
  uint32_t *s_cur = s_mem;                   // [TX] next free slot of each tile
  uint32_t *s_pre = s_cur + TX;              // [VW][TP] first slot of each group
  uint32_t *s_mask = s_pre + VW * TP;        // [2][VW][TP]
  __shared__ uint32_t s_longest;             // longest of the tile row's lists (chunk 0)
  if (threadIdx.x == 0) s_longest = 0u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t tile0 = uint32_t(cam.tile_base) + uint32_t(grow - cam.trow_base) * uint32_t(TX);
  {
    // per tile column: instances of the whole tile row and of the earlier chunks
    const uint32_t cb = P.chunk_base[grow], nch = P.chunk_base[grow + 1] - cb;
    uint32_t *s_tot = s_pre, *s_bef = s_pre + TX;  // 2 TX words of the group-prefix buffer
    for (int x = threadIdx.x; x < TX; x += NT) {
      uint32_t tot = 0, bef = 0;
      for (uint32_t k = 0; k < nch; ++k) {
        const uint32_t n = P.cnt2[size_t(cb + k) * size_t(P.max_tiles_x) + x];
        tot += n;
        bef += k < uint32_t(chunk_c) ? n : 0u;
      }
      s_tot[x] = tot;
      s_bef[x] = bef;
    }
    __syncthreads();
    __shared__ uint32_t s_ws[33];
    const int per = (TX + NT - 1) / NT;
    const int x0 = min(TX, int(threadIdx.x) * per), x1 = min(TX, x0 + per);
    uint32_t csum = 0;
    for (int x = x0; x < x1; ++x) csum += s_tot[x];
    uint32_t ctot;
    const uint32_t cpre = block_excl_scan(csum, s_ws, &ctot);  // instances before the column chunk
    const unsigned long long base = P.trow_inst[grow];
    uint32_t o = uint32_t(min(base, (unsigned long long)P.cap)) + cpre, longest = 0;
    for (int j = 0; j < per; ++j) {
      const int x = x0 + j;
      const bool in = x < x1;
      const uint32_t n = in ? s_tot[x] : 0u;
      if (in) s_cur[x] = o + s_bef[x];
      if (chunk_c == 0) {
        const uint2 r = make_uint2(min(o, P.cap), min(o + n, P.cap));
        if (in) P.ranges[tile0 + x] = r;
        if (P.class_tiles) {  // one atomic per class and warp: of 518,400 tiles one by one they took 260 us
          longest = max(longest, r.y - r.x);
          const int c = in ? tile_class_of(r.y - r.x) : kTileClasses;
          const uint32_t peers = __match_any_sync(0xffffffffu, c);
          uint32_t at = 0;
          if (in && lane == __ffs(peers) - 1) at = atomicAdd(&P.counters->tile_class[c], __popc(peers));
          at = __shfl_sync(0xffffffffu, at, __ffs(peers) - 1) + __popc(peers & lt);
          if (in) P.class_tiles[size_t(c) * size_t(P.tiles) + at] = tile0 + x;
        }
      }
      o += n;
    }
    longest = __reduce_max_sync(0xffffffffu, longest);
    if (lane == 0 && longest) atomicMax(&s_longest, longest);
  }
  __syncthreads();
  if (threadIdx.x == 0 && s_longest) atomicMax(&P.counters->longest, s_longest);
  for (int j = threadIdx.x; j < 2 * VW * TP; j += NT) s_mask[j] = 0u;
  constexpr uint32_t STEP = uint32_t(NT) * KR;
  uint2 nxt[KR];
  uint32_t nxt_e[KR];  // first partial-sum slot of each row (plans with the backward)
  auto load_rows = [&](uint32_t base) {
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const uint32_t i = base + uint32_t(k * NT) + threadIdx.x;
      nxt[k] = i < rr.y ? P.rows[i] : make_uint2(0u, 0u);
      if (P.inst_e && i < rr.y) {
        const uint2 re = P.row_e[i];
        nxt_e[k] = P.e_base[re.x] + re.y;
      }
    }
  };
  if (rr.x < rr.y) load_rows(rr.x);
  int buf = 0;
  for (uint32_t base = rr.x; base < rr.y; base += STEP) {
    uint2 cur[KR];
    uint32_t cur_e[KR];
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      cur[k] = nxt[k];
      cur_e[k] = nxt_e[k];
    }
    if (base + STEP < rr.y) load_rows(base + STEP);
    uint32_t *mask = s_mask + buf * VW * TP;
    __syncthreads();  // masks of this buffer cleared; the previous step's reads are done
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const int g = k * (NT / 32) + warp;
      const uint2 cl = row_cols(cur[k].y, uint32_t(TX));
      const uint32_t xa = cl.x, len = cl.y;
      for (uint32_t t = 0; t < len; ++t) atomicOr(&mask[g * TP + int(xa + t)], 1u << lane);
    }
    __syncthreads();
    // per tile (one thread each), the group counts in group order
    uint32_t *other = s_mask + (1 - buf) * VW * TP;
    for (int x = threadIdx.x; x < TX; x += NT) {
      uint32_t run = s_cur[x];
#pragma unroll 8
      for (int g = 0; g < VW; ++g) {
        s_pre[g * TP + x] = run;
        run += __popc(mask[g * TP + x]);
        other[g * TP + x] = 0u;
      }
      s_cur[x] = run;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const int g = k * (NT / 32) + warp;
      const uint2 cl = row_cols(cur[k].y, uint32_t(TX));
      const uint32_t xa = cl.x, len = cl.y;
      for (uint32_t t = 0; t < len; ++t) {
        const int x = int(xa + t);
        const uint32_t dst = s_pre[g * TP + x] + __popc(mask[g * TP + x] & lt);
        if (dst < P.cap) {
          P.inst[dst] = cur[k].x;
          if (P.inst_e) P.inst_e[dst] = cur_e[k] + t;
        }
      }
    }
    buf = 1 - buf;
  }
}

template <int NT, int KR>
static size_t list_smem(int max_tiles_x) {
  return sizeof(uint32_t) * size_t(max_tiles_x + 1) * size_t(1 + 3 * (NT / 32) * KR);
}

// Rows per chunk: the shortest power of two from 512 to 8,192 that leaves fewer than 16 chunks
// per SM (chosen on the device, trow_plan_kernel): long lists amortise a chunk's prologue (the
// counts of all the tile row's chunks), short ones still occupy every SM.  A 720p frame's 0.43 M
// rows in chunks of 512: 17 us, against 39 us in chunks of 8,192 (90 of them).  Longer when the
// per-chunk column counts would pass 32 M entries.
// With a shortest chunk of a row per tile column at least, the column counts take no more than 4 bytes
// per unit of capacity, on views wider than 512 tiles too (at 512 rows up to 32 bytes): where the
// workspace is short.  It costs time there (32768x512, 50k primitives: binning 147 against 128 us).
uint32_t list_rows_short(int max_tiles_x) {
  uint32_t cr = kListRowsLo;
  while (cr < uint32_t(max_tiles_x)) cr <<= 1;
  return cr;
}
uint32_t list_rows_hi(int64_t cap, int max_tiles_x) {
  uint32_t cr = 8192;
  while ((uint64_t(cap) / cr) * uint64_t(max_tiles_x) > (uint64_t(32) << 20)) cr <<= 1;
  return cr;
}
uint32_t list_target(int num_sms) { return uint32_t(num_sms) * 16; }
uint64_t list_max_chunks(int64_t trows, int64_t cap, int max_tiles_x, int num_sms, uint32_t rows_lo) {
  const uint64_t by_lo = uint64_t(cap) / rows_lo, by_hi = uint64_t(cap) / list_rows_hi(cap, max_tiles_x);
  return uint64_t(trows) + std::min<uint64_t>(by_lo, std::max<uint64_t>(list_target(num_sms), by_hi)) + 1;
}

cudaError_t launch_lists(const ListParams &P, int num_sms, cudaStream_t st) {
  if (P.trows == 0) return cudaSuccess;
  const unsigned cg = unsigned(std::min<uint64_t>(P.max_chunks, uint64_t(num_sms) * 8));
  launch(list_count_kernel, cg, 256, sizeof(uint32_t) * size_t(P.max_tiles_x + 1), st, P);
  constexpr size_t kBudget = 200 * 1024;
  auto run = [&](auto kernel, int nt, size_t smem) -> cudaError_t {
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
      if (e != cudaSuccess) return e;
    }
    launch(kernel, P.max_chunks, nt, smem, st, P);
    return cudaGetLastError();
  };
  const int mtx = P.max_tiles_x;
  if (list_smem<256, 4>(mtx) <= kBudget) return run(list_kernel<256, 4>, 256, list_smem<256, 4>(mtx));
  if (list_smem<256, 1>(mtx) <= kBudget) return run(list_kernel<256, 1>, 256, list_smem<256, 1>(mtx));
  return run(list_kernel<128, 1>, 128, list_smem<128, 1>(mtx));
}

}  // namespace raygs
