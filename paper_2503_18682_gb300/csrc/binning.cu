// Binning for the depth order of Eq. rendering.
//
//   1. Stable LSD radix sort of the visible (primitive, view) pairs by float32 centre
//      depth.  The first pass reads the dense per-(view, primitive) key array, drops
//      culled entries and materialises the pair index as the value, so ties keep the
//      primitive order within a view; the last pass leaves each pair's tile rows in place
//      of its key.
//   2. With several views, one more stable pass by view: the pairs view by view, each view in
//      depth order, with their ids and their positions in the depth order.
//   3. Support rows (rows.cu): each pair -> the tile rows of its screen rectangle, each row
//      -> the run of tiles whose pixel centres can meet the pair's support, placed into
//      per-tile-row lists in depth order.
//   4. Per tile row, in chunks of rows: the rows expanded into per-tile instance lists in
//      depth order, and the per-tile [start, end) ranges.
//
// The radix sort is reduce-then-scan (upsweep histogram, one scan CTA per digit, downsweep
// scatter) with persistent CTAs that own contiguous tile ranges: no CTA ever waits on
// another.  The upsweep counts runs of equal digits per thread; ranking inside a tile is
// stable (warp multi-split by digit-bit ballots + per-warp counters) and the scatter goes
// through shared memory so that global writes are coalesced runs.
#include "bins.cuh"

namespace raygs {

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortIPT = 8;
constexpr int kSortTile = kSortThreads * kSortIPT;  // 2048 items
constexpr int kSortNoScan = 16;  // CTAs up to which a pass needs no scan kernel

__device__ __forceinline__ void cta_tiles(uint32_t count, uint32_t &lo, uint32_t &hi) {
  uint32_t ntiles = (count + kSortTile - 1) / kSortTile;
  uint32_t t0 = uint32_t((uint64_t(ntiles) * blockIdx.x) / gridDim.x);
  uint32_t t1 = uint32_t((uint64_t(ntiles) * (blockIdx.x + 1)) / gridDim.x);
  lo = t0 * kSortTile;
  hi = min(t1 * uint32_t(kSortTile), count);
  if (lo > hi) lo = hi;
}

__device__ __forceinline__ uint32_t pass_count(const SortPass &p) {
  return p.d_count ? min(*p.d_count, p.count_max) : p.count_max;
}

// Digit histogram of the CTA's items.  Each thread counts 16 consecutive keys as runs of
// equal digits (the tile-id passes see long runs: instances come in depth order, tile rows
// in order) and adds each run once to its warp's shared histogram.
template <int BITS, bool FILTER>
__global__ void __launch_bounds__(kSortThreads) sort_upsweep(SortPass p) {
  constexpr int R = 1 << BITS;
  constexpr int KPT = 16;  // keys per thread per step
  __shared__ uint32_t h[kSortWarps][R];
  for (int i = threadIdx.x; i < kSortWarps * R; i += kSortThreads) (&h[0][0])[i] = 0;
  __syncthreads();
  uint32_t lo, hi;
  cta_tiles(pass_count(p), lo, hi);
  const int warp = threadIdx.x >> 5;
  for (uint32_t base = lo; base < hi; base += kSortThreads * KPT) {
    const uint32_t i0 = base + threadIdx.x * KPT;
    uint32_t k[KPT];
    if (i0 + KPT <= hi) {
#pragma unroll
      for (int q = 0; q < KPT / 4; ++q) {
        const uint4 v = *reinterpret_cast<const uint4 *>(p.keys_in + i0 + 4 * q);
        k[4 * q] = v.x; k[4 * q + 1] = v.y; k[4 * q + 2] = v.z; k[4 * q + 3] = v.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < KPT; ++j) k[j] = i0 + j < hi ? p.keys_in[i0 + j] : kCulled;
    }
    uint32_t cur = 0xFFFFFFFFu, cnt = 0;
#pragma unroll
    for (int j = 0; j < KPT; ++j) {
      const bool valid = i0 + j < hi && !(FILTER && k[j] == kCulled);
      if (!valid) continue;
      const uint32_t d = (k[j] >> p.shift) & (R - 1);
      if (d == cur) {
        ++cnt;
      } else {
        if (cnt) atomicAdd(&h[warp][cur], cnt);
        cur = d;
        cnt = 1;
      }
    }
    if (cnt) atomicAdd(&h[warp][cur], cnt);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < R; d += kSortThreads) {
    uint32_t s = 0;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) s += h[w][d];
    p.hist[size_t(d) * p.G + blockIdx.x] = s;
  }
}

// MODE: what a pass does with its payloads.  First drops the culled keys and packs the tile
// rows beside key and id, last unpacks them (see SortPass), split also writes the items'
// indices; compiled apart, so that the plain passes keep their 64 registers.
enum SortMode { kSortPlain = 0, kSortFirst = 1, kSortLast = 2, kSortSplit = 3 };

template <int BITS, int MODE>
__global__ void __launch_bounds__(kSortThreads, 4) sort_downsweep(SortPass p) {
  constexpr int R = 1 << BITS;
  __shared__ uint32_t s_keys[kSortTile];
  __shared__ uint32_t s_vals[kSortTile];
  __shared__ uint32_t s_ids[MODE == kSortSplit ? kSortTile : 1];
  __shared__ uint32_t s_cnt[kSortWarps][R];
  __shared__ uint32_t s_base[R];
  __shared__ uint32_t s_tpre[R];
  __shared__ uint32_t s_tot[R];
  __shared__ uint32_t s_ws[33];

  uint32_t lo, hi;
  cta_tiles(pass_count(p), lo, hi);
  {  // first output of each digit: the lower digits' items, then the lower CTAs' of this digit
    static_assert(R <= kSortThreads, "one digit per thread");
    uint32_t before = 0, total = 0;
    if (threadIdx.x < R) {
      const uint32_t *row = p.hist + size_t(threadIdx.x) * p.G;
      if (p.G > kSortNoScan) {
        before = row[blockIdx.x];
        total = p.digit_total[threadIdx.x];
      } else {
        for (int c = 0; c < p.G; ++c) {
          const uint32_t n = row[c];
          total += n;
          before += c < int(blockIdx.x) ? n : 0u;
        }
      }
    }
    uint32_t all;
    const uint32_t lower = block_excl_scan(total, s_ws, &all);
    if (p.G <= kSortNoScan && blockIdx.x == 0 && threadIdx.x < R) p.digit_total[threadIdx.x] = total;
    if (threadIdx.x < R) s_base[threadIdx.x] = lower + before;
    if (p.d_total && blockIdx.x == 0 && threadIdx.x == 0) *p.d_total = all;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;

  // the keys and values of the next tile are loaded while the current one is ranked
  uint32_t nkey[kSortIPT], nval[kSortIPT];
  auto load = [&](uint32_t base) {
#pragma unroll
    for (int r = 0; r < kSortIPT; ++r) {
      const uint32_t idx = base + warp * (32 * kSortIPT) + r * 32 + lane;
      nkey[r] = idx < hi ? p.keys_in[idx] : 0u;
      nval[r] = MODE == kSortFirst ? idx : (idx < hi ? p.vals_in[idx] : 0u);
    }
  };
  if (lo < hi) load(lo);
  for (uint32_t base = lo; base < hi; base += kSortTile) {
    for (int i = threadIdx.x; i < kSortWarps * R; i += kSortThreads) (&s_cnt[0][0])[i] = 0;
    uint32_t key[kSortIPT], val[kSortIPT], off[kSortIPT];
#pragma unroll
    for (int r = 0; r < kSortIPT; ++r) {
      key[r] = nkey[r];
      val[r] = nval[r];
    }
    if (base + kSortTile < hi) load(base + kSortTile);
    __syncthreads();
    uint32_t vmask = 0;
#pragma unroll
    for (int r = 0; r < kSortIPT; ++r) {
      const uint32_t idx = base + warp * (32 * kSortIPT) + r * 32 + lane;
      const bool ok = idx < hi;
      const uint32_t k = key[r];
      const bool valid = ok && !(MODE == kSortFirst && k == kCulled);
      uint32_t d = (k >> p.shift) & (R - 1);
      // lanes holding the same digit: one ballot per digit bit (warp-level multi-split)
      uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
      for (int bit = 0; bit < BITS; ++bit) {
        const uint32_t bal = __ballot_sync(0xffffffffu, (d >> bit) & 1u);
        peers &= ((d >> bit) & 1u) ? bal : ~bal;
      }
      if (!valid) peers = 1u << lane;
      uint32_t c = valid ? s_cnt[warp][d] : 0u;
      __syncwarp();
      if (valid && lane == 31 - __clz(peers)) s_cnt[warp][d] = c + __popc(peers);
      __syncwarp();
      off[r] = c + __popc(peers & lt);
      vmask |= valid ? (1u << r) : 0u;
    }
    __syncthreads();
    for (int d = threadIdx.x; d < R; d += kSortThreads) {
      uint32_t run = 0;
#pragma unroll
      for (int w = 0; w < kSortWarps; ++w) {
        uint32_t c = s_cnt[w][d];
        s_cnt[w][d] = run;
        run += c;
      }
      s_tot[d] = run;
    }
    __syncthreads();
    {
      constexpr int PER = (R + kSortThreads - 1) / kSortThreads;
      uint32_t loc[PER];
      uint32_t s = 0;
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        int d = threadIdx.x * PER + j;
        loc[j] = d < R ? s_tot[d] : 0u;
        s += loc[j];
      }
      uint32_t tot;
      uint32_t run = block_excl_scan(s, s_ws, &tot);
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        int d = threadIdx.x * PER + j;
        if (d < R) s_tpre[d] = run;
        run += loc[j];
      }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortIPT; ++r) {
      if (vmask & (1u << r)) {
        uint32_t d = (key[r] >> p.shift) & (R - 1);
        uint32_t pos = s_tpre[d] + s_cnt[warp][d] + off[r];
        s_keys[pos] = key[r];
        s_vals[pos] = val[r];
        if (MODE == kSortSplit) s_ids[pos] = base + warp * (32 * kSortIPT) + r * 32 + lane;
      }
    }
    __syncthreads();
    const uint32_t nvalid = s_tpre[R - 1] + s_tot[R - 1];
    for (uint32_t j = threadIdx.x; j < nvalid; j += kSortThreads) {
      uint32_t k = s_keys[j];
      uint32_t d = (k >> p.shift) & (R - 1);
      uint32_t dst = s_base[d] + j - s_tpre[d];
      uint32_t kout = k, vout = s_vals[j];
      if (MODE == kSortFirst) {  // its consumed digit makes room for the tile rows
        const uint32_t ri = p.row_info[vout], cnt = ri >> 8;
        kout = (k & ~0xFFu) | (ri & 0xFFu);
        if (p.id_bits < 32) {
          const uint32_t field = 0xFFFFFFFFu >> p.id_bits;
          vout |= (cnt < 255u && cnt < field ? cnt : field) << p.id_bits;
        }
      } else if (MODE == kSortLast) {  // tile rows and view as key, the bare id
        const bool packed = p.id_bits < 32;
        const uint32_t field = packed ? 0xFFFFFFFFu >> p.id_bits : 0u;
        uint32_t ty0 = k & 0xFFu, cnt = packed ? vout >> p.id_bits : 0u;
        if (packed) vout &= (1u << p.id_bits) - 1u;
        if (cnt >= field || ty0 == 255u) {
          const uint2 r = p.row_rect[vout];
          ty0 = r.x >> 16;
          cnt = (r.y >> 16) - ty0 + 1;
        }
        kout = ty0 | ((cnt - 1u) << 12) | ((vout / p.n) << 24);
      }
      p.keys_out[dst] = kout;
      p.vals_out[dst] = vout;
      if (MODE == kSortSplit) p.index_out[dst] = s_ids[j];
    }
    __syncthreads();
    for (int d = threadIdx.x; d < R; d += kSortThreads) s_base[d] += s_tot[d];
    __syncthreads();
  }
}

// Exclusive scan of one digit's counts over the CTAs, in place, and the digit's total (one
// CTA per digit); the downsweep scans the R digit totals itself.
constexpr int kSortMaxGrid = 1024;

__global__ void __launch_bounds__(256) hist_scan_kernel(uint32_t *hist, int G, uint32_t *digit_total) {
  __shared__ uint32_t ws[33];
  constexpr int PER = kSortMaxGrid / 256;
  uint32_t *row = hist + size_t(blockIdx.x) * G;
  uint32_t v[PER], s = 0;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = threadIdx.x * PER + j;
    v[j] = i < G ? row[i] : 0u;
    s += v[j];
  }
  uint32_t tot;
  uint32_t run = block_excl_scan(s, ws, &tot);
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = threadIdx.x * PER + j;
    if (i < G) row[i] = run;
    run += v[j];
  }
  if (threadIdx.x == 0) digit_total[blockIdx.x] = tot;
}

// One LSD pass: 8-bit digits for the depth sort, 4 or 6 bits for the split by view.  The grid
// is at most one CTA per 2,048 items.  Up to kSortNoScan CTAs (32,768 items) every downsweep
// CTA reads the counts of all of them instead of a scan kernel's offsets: two launches instead
// of three; the 720p frame's 500,000 pairs (245 CTAs) are past the point where that reading
// costs more than the launch.
template <int BITS, int MODE>
static cudaError_t sort_pass(const SortPass &p, cudaStream_t st) {
  sort_upsweep<BITS, MODE == kSortFirst><<<p.G, kSortThreads, 0, st>>>(p);
  if (p.G > kSortNoScan) hist_scan_kernel<<<1 << BITS, 256, 0, st>>>(p.hist, p.G, p.digit_total);
  sort_downsweep<BITS, MODE><<<p.G, kSortThreads, 0, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_sort_pass(SortPass p, cudaStream_t st) {
  const uint32_t need = (p.count_max + uint32_t(kSortTile) - 1u) / uint32_t(kSortTile);  // CTAs with work
  p.G = need < uint32_t(p.G) ? (need ? int(need) : 1) : p.G;
  if (p.row_info) return sort_pass<8, kSortFirst>(p, st);
  if (p.row_rect) return sort_pass<8, kSortLast>(p, st);
  if (!p.index_out) return sort_pass<8, kSortPlain>(p, st);
  return p.n_views <= 16 ? sort_pass<4, kSortSplit>(p, st) : sort_pass<6, kSortSplit>(p, st);
}

// ------------------------------------------------- tile rows -> per-tile instance lists
__device__ __forceinline__ const DevCam &view_of_trow(const ExpandParams &E, int grow, int &v_out) {
  int v = 0;
  while (v + 1 < E.n_views && E.cams[v + 1].trow_base <= grow) ++v;
  v_out = v;
  return E.cams[v];
}

// Exclusive scan of the per-tile-row instance totals in place (one block, 64-bit running
// sums): each tile row's first instance, the instance total, its capacity clamp and the
// overflow flag.
__global__ void __launch_bounds__(1024) trow_scan_kernel(unsigned long long *v, int n, Counters *c, uint32_t cap) {
  __shared__ unsigned long long ws[32];
  const int per = (n + 1023) / 1024;
  const int b = min(n, int(threadIdx.x) * per), e = min(n, b + per);
  unsigned long long s = 0;
  for (int i = b; i < e; ++i) s += v[i];
  // block exclusive scan of s (warp scans of 64-bit values, then of the warp totals)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[warp] = x;
  __syncthreads();
  if (warp == 0) {
    unsigned long long t = ws[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    ws[lane] = t;
  }
  __syncthreads();
  unsigned long long run = (warp ? ws[warp - 1] : 0ull) + x - s;
  for (int i = b; i < e; ++i) {
    const unsigned long long t = v[i];
    v[i] = run;
    run += t;
  }
  if (threadIdx.x == 1023) {
    const unsigned long long total = ws[31];
    c->n_instances = total;
    c->n_inst_clamped = total > cap ? cap : uint32_t(total);
    if (total > cap) c->overflow = 1u;
  }
}

// Instance lists of one tile row.  Rows are taken in sorted (depth) order, NT * KR at a
// time, in 32-row groups (KR * NT / 32 groups: row q of the step is lane q % 32 of group
// q / 32); every lane marks the tiles of its row in its group's bit mask per tile, and the
// rank of (row, tile) is the tile's running cursor plus the rows of lower groups and lower
// lanes that cover the same tile.  Each tile's list keeps depth order.  The masks are
// double-buffered (the buffer of the next step is cleared while this one is read) and the
// rows of the next step are loaded during this one.
// The chunk of rows a CTA owns: tile row t (largest t with chunk_base[t] <= chunk) and its
// rows [first, last).
__device__ __forceinline__ bool chunk_of(const ExpandParams &E, uint32_t chunk, int &t, int &c, uint2 &rows) {
  if (chunk >= E.chunk_base[E.trows]) return false;
  int lo = 0, hi = E.trows - 1;
  while (lo < hi) {
    const int m = (lo + hi + 1) >> 1;
    if (E.chunk_base[m] <= chunk) lo = m; else hi = m - 1;
  }
  t = lo;
  c = int(chunk - E.chunk_base[t]);
  const uint2 rr = E.trow_ranges[t];
  const uint32_t first = rr.x + uint32_t(c) * uint32_t(E.chunk_rows);
  rows = make_uint2(min(first, rr.y), min(first + uint32_t(E.chunk_rows), rr.y));
  return true;
}

// Chunks per tile row (at least one) and their exclusive scan (one block).
__global__ void __launch_bounds__(1024) chunk_scan_kernel(ExpandParams E) {
  __shared__ uint32_t ws[33];
  const int per = (E.trows + 1023) / 1024;
  const int b = min(E.trows, int(threadIdx.x) * per), e = min(E.trows, b + per);
  auto nchunks = [&](int t) {
    const uint2 rr = E.trow_ranges[t];
    const uint32_t n = rr.y - rr.x;
    return n == 0 ? 1u : (n + uint32_t(E.chunk_rows) - 1) / uint32_t(E.chunk_rows);
  };
  uint32_t s = 0;
  for (int t = b; t < e; ++t) s += nchunks(t);
  uint32_t tot;
  uint32_t run = block_excl_scan(s, ws, &tot);
  for (int t = b; t < e; ++t) {
    E.chunk_base[t] = run;
    run += nchunks(t);
  }
  if (threadIdx.x == 0) E.chunk_base[E.trows] = min(tot, uint32_t(E.max_chunks));
}

// Instances per tile column of one chunk: each row covers the tile columns
// [txa, txa + len); a difference array over the columns and its prefix sum count them.
__global__ void __launch_bounds__(256) chunk_count_kernel(ExpandParams E) {
  extern __shared__ uint32_t s_diff[];  // [max_tiles_x + 1]
  __shared__ uint32_t s_ws[33];
  int t, c;
  uint2 rows;
  if (!chunk_of(E, blockIdx.x, t, c, rows)) return;
  int v;
  const DevCam &cam = view_of_trow(E, t, v);
  const int TX = cam.tiles_x;
  for (int x = threadIdx.x; x <= TX; x += blockDim.x) s_diff[x] = 0u;
  __syncthreads();
  // four rows per thread at a time, their loads issued before any of their atomics
  for (uint32_t i0 = rows.x + threadIdx.x; i0 < rows.y; i0 += 4 * blockDim.x) {
    uint32_t pk[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t i = i0 + k * blockDim.x;
      pk[k] = i < rows.y ? E.rows[i].y : 0u;  // 0: no tiles
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (pk[k] >> 16) {
        atomicAdd(&s_diff[pk[k] & 0xFFFFu], 1u);
        atomicSub(&s_diff[(pk[k] & 0xFFFFu) + (pk[k] >> 16)], 1u);
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
  uint32_t *out = E.chunk_cnt + size_t(blockIdx.x) * size_t(E.max_tiles_x);
  unsigned long long mine = 0;
  for (int x = x0; x < x1; ++x) {
    run += s_diff[x];
    out[x] = run;
    mine += run;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0 && mine) atomicAdd(&E.trow_base[t], mine);
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
__global__ void __launch_bounds__(NT) expand_kernel(ExpandParams E) {
  constexpr int VW = NT / 32 * KR;  // row groups per step
  extern __shared__ uint32_t s_mem[];
  int grow, chunk_c;
  uint2 rr;
  if (!chunk_of(E, blockIdx.x, grow, chunk_c, rr)) return;
  int v;
  const DevCam &cam = view_of_trow(E, grow, v);
  const int TX = cam.tiles_x;
  const int TP = TX | 1;                     // odd row stride: no bank conflicts down a column
  uint32_t *s_cur = s_mem;                   // [TX] next free slot of each tile
  uint32_t *s_pre = s_cur + TX;              // [VW][TP] first slot of each group
  uint32_t *s_mask = s_pre + VW * TP;        // [2][VW][TP]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t tile0 = uint32_t(cam.tile_base) + uint32_t(grow - cam.trow_base) * uint32_t(TX);
  {
    // per tile column: instances of the whole tile row and of the earlier chunks
    const uint32_t cb = E.chunk_base[grow], nch = E.chunk_base[grow + 1] - cb;
    uint32_t *s_tot = s_pre, *s_bef = s_pre + TX;  // 2 TX words of the group-prefix buffer
    for (int x = threadIdx.x; x < TX; x += NT) {
      uint32_t tot = 0, bef = 0;
      for (uint32_t k = 0; k < nch; ++k) {
        const uint32_t n = E.chunk_cnt[size_t(cb + k) * size_t(E.max_tiles_x) + x];
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
    const unsigned long long base = E.trow_base[grow];
    uint32_t o = uint32_t(min(base, (unsigned long long)E.cap)) + cpre;
    for (int x = x0; x < x1; ++x) {
      const uint32_t n = s_tot[x];
      s_cur[x] = o + s_bef[x];
      if (chunk_c == 0) E.ranges[tile0 + x] = make_uint2(min(o, E.cap), min(o + n, E.cap));
      o += n;
    }
  }
  __syncthreads();
  for (int j = threadIdx.x; j < 2 * VW * TP; j += NT) s_mask[j] = 0u;
  constexpr uint32_t STEP = uint32_t(NT) * KR;
  uint2 nxt[KR];
  uint32_t nxt_e[KR];  // first partial-sum slot of each row (plans with the backward)
  auto load_rows = [&](uint32_t base) {
#pragma unroll
    for (int k = 0; k < KR; ++k) {
      const uint32_t i = base + uint32_t(k * NT) + threadIdx.x;
      nxt[k] = i < rr.y ? E.rows[i] : make_uint2(0u, 0u);
      if (E.inst_e && i < rr.y) {
        const uint2 re = E.row_e[i];
        nxt_e[k] = E.e_base[re.x] + re.y;
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
      const uint32_t xa = cur[k].y & 0xFFFFu, len = cur[k].y >> 16;
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
      const uint32_t xa = cur[k].y & 0xFFFFu, len = cur[k].y >> 16;
      for (uint32_t t = 0; t < len; ++t) {
        const int x = int(xa + t);
        const uint32_t dst = s_pre[g * TP + x] + __popc(mask[g * TP + x] & lt);
        if (dst < E.cap) {
          E.inst[dst] = cur[k].x;
          if (E.inst_e) E.inst_e[dst] = cur_e[k] + t;
        }
      }
    }
    buf = 1 - buf;
  }
}

template <int NT, int KR>
size_t expand_smem(int max_tiles_x) {
  return sizeof(uint32_t) * size_t(max_tiles_x + 1) * size_t(1 + 3 * (NT / 32) * KR);
}


int expand_chunk_rows(int64_t cap, int max_tiles_x) {
  // 8192 rows per chunk, more when the per-chunk column counts would pass 32 M entries
  int64_t ch = 8192;
  const int64_t need = (cap * int64_t(max_tiles_x > 0 ? max_tiles_x : 1)) / (int64_t(32) << 20) + 1;
  if (need > ch) ch = need;
  return int(ch > (int64_t(1) << 30) ? (int64_t(1) << 30) : ch);
}

int64_t expand_max_chunks(int64_t trows, int64_t cap, int chunk_rows) {
  return trows + cap / chunk_rows + 1;
}

cudaError_t launch_expand(const ExpandParams &E, cudaStream_t st) {
  if (E.trows == 0) return cudaSuccess;
  chunk_scan_kernel<<<1, 1024, 0, st>>>(E);
  chunk_count_kernel<<<E.max_chunks, 256, sizeof(uint32_t) * size_t(E.max_tiles_x + 1), st>>>(E);
  trow_scan_kernel<<<1, 1024, 0, st>>>(E.trow_base, E.trows, E.counters, E.cap);
  constexpr size_t kBudget = 200 * 1024;
  auto run = [&](auto kernel, int nt, size_t smem) -> cudaError_t {
    if (smem > 48 * 1024) {
      cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
      if (e != cudaSuccess) return e;
    }
    kernel<<<E.max_chunks, nt, smem, st>>>(E);
    return cudaGetLastError();
  };
  const int mtx = E.max_tiles_x;
  if (expand_smem<256, 4>(mtx) <= kBudget) return run(expand_kernel<256, 4>, 256, expand_smem<256, 4>(mtx));
  if (expand_smem<256, 1>(mtx) <= kBudget) return run(expand_kernel<256, 1>, 256, expand_smem<256, 1>(mtx));
  return run(expand_kernel<128, 1>, 128, expand_smem<128, 1>(mtx));
}

}  // namespace raygs
