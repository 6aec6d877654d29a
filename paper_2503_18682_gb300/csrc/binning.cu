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
//   4. Per tile row (lists.cu): the rows expanded into per-tile instance lists in depth order,
//      and the per-tile [start, end) ranges.
//
// This file holds the radix sort.  It is reduce-then-scan (upsweep histogram, one scan CTA per digit, downsweep
// scatter), with persistent CTAs that own contiguous tile ranges: no CTA ever waits on
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
// equal digits (the top digit of a depth is little more than its exponent, and the views are few:
// long runs) and adds each run once to its warp's shared histogram.
template <int BITS, bool FILTER>
__global__ void __launch_bounds__(kSortThreads) sort_upsweep(SortPass p) {
  await_previous();
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
// indices; compiled apart, so that the plain passes keep their 64 registers (the first and
// the last pass spill 16 bytes at that bound, the split by up to 16 views 68, by more 48).
enum SortMode { kSortPlain = 0, kSortFirst = 1, kSortLast = 2, kSortSplit = 3 };

template <int BITS, int MODE>
__global__ void __launch_bounds__(kSortThreads, 4) sort_downsweep(SortPass p) {
  await_previous();
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
  await_previous();
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

// The whole depth sort of up to 6,144 pairs in one CTA: the keys of the pairs that are left (ids fit
// 16 bits) stay in shared memory between the four passes, ranked as in sort_downsweep, each warp
// over a contiguous part.  Bound by the latency of its steps: a frame of
// 1,000 primitives took 92 us with the eight launches of the passes and 75 us with this one, of 4,096
// 132 and 121, of 6,000 155 and 149; at 8,192 (16 items per thread) both took 173.
constexpr int kSmallThreads = 512, kSmallWarps = kSmallThreads / 32, kSmallIPT = 12;
constexpr int kSmallItems = kSmallThreads * kSmallIPT;
constexpr size_t kSmallSmem = size_t(kSmallItems) * 6 + size_t(kSmallWarps) * 256 * 4;

__global__ void __launch_bounds__(kSmallThreads) sort_small_kernel(SortPass p) {
  await_previous();
  extern __shared__ uint32_t s_small[];
  uint32_t *s_key = s_small;                                               // [kSmallItems]
  uint32_t(*s_cnt)[256] = reinterpret_cast<uint32_t(*)[256]>(s_key + kSmallItems);  // [kSmallWarps][256]
  uint16_t *s_id = reinterpret_cast<uint16_t *>(s_cnt + kSmallWarps);      // [kSmallItems]
  __shared__ uint32_t s_base[256];
  __shared__ uint32_t s_ws[33];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t m = min(p.count_max, uint32_t(kSmallItems));  // items before the pass
  for (int shift = 0; shift < 32; shift += 8) {
    const uint32_t rounds = (m + kSmallThreads - 1) / kSmallThreads, first = warp * (32 * rounds) + lane;
    uint32_t key[kSmallIPT], id[kSmallIPT], off[kSmallIPT], vmask = 0;
#pragma unroll
    for (int r = 0; r < kSmallIPT; ++r) {
      const uint32_t idx = first + r * 32;
      const bool ok = r < rounds && idx < m;
      key[r] = !ok ? kCulled : shift ? s_key[idx] : p.keys_in[idx];
      id[r] = !ok ? 0u : shift ? s_id[idx] : idx;
      if (ok && (shift || key[r] != kCulled)) vmask |= 1u << r;
    }
    for (int i = threadIdx.x; i < kSmallWarps * 256; i += kSmallThreads) (&s_cnt[0][0])[i] = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallIPT; ++r) {
      if (r >= rounds) break;
      const bool valid = (vmask >> r) & 1u;
      const uint32_t d = (key[r] >> shift) & 255u;
      uint32_t peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
      for (int bit = 0; bit < 8; ++bit) {
        const uint32_t bal = __ballot_sync(0xffffffffu, (d >> bit) & 1u);
        peers &= ((d >> bit) & 1u) ? bal : ~bal;
      }
      if (!valid) peers = 1u << lane;
      const uint32_t c = valid ? s_cnt[warp][d] : 0u;
      __syncwarp();
      if (valid && lane == 31 - __clz(peers)) s_cnt[warp][d] = c + __popc(peers);
      __syncwarp();
      off[r] = c + __popc(peers & lt);
    }
    __syncthreads();
    uint32_t run = 0;
    if (threadIdx.x < 256) {
#pragma unroll
      for (int w = 0; w < kSmallWarps; ++w) {
        const uint32_t c = s_cnt[w][threadIdx.x];
        s_cnt[w][threadIdx.x] = run;
        run += c;
      }
    }
    uint32_t kept;
    const uint32_t lower = block_excl_scan(run, s_ws, &kept);
    if (threadIdx.x < 256) s_base[threadIdx.x] = lower;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallIPT; ++r) {
      if (vmask & (1u << r)) {
        const uint32_t d = (key[r] >> shift) & 255u, pos = s_base[d] + s_cnt[warp][d] + off[r];
        s_key[pos] = key[r];
        s_id[pos] = uint16_t(id[r]);
      }
    }
    m = kept;
    __syncthreads();
  }
  for (uint32_t j = threadIdx.x; j < m; j += kSmallThreads) {
    const uint32_t v = s_id[j], ri = p.row_info[v];
    uint32_t ty0 = ri & 0xFFu, cnt = ri >> 8;
    if (cnt >= 255u || ty0 == 255u) {
      const uint2 r = p.row_rect[v];
      ty0 = r.x >> 16;
      cnt = (r.y >> 16) - ty0 + 1;
    }
    p.keys_out[j] = ty0 | ((cnt - 1u) << 12) | ((v / p.n) << 24);
    p.vals_out[j] = v;
  }
  if (threadIdx.x == 0) *p.d_total = m;
}

bool sort_is_small(uint64_t pairs) { return pairs <= uint64_t(kSmallItems); }

cudaError_t launch_sort_small(const SortPass &p, cudaStream_t st) {
  cudaError_t e = cudaFuncSetAttribute(sort_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kSmallSmem));
  if (e != cudaSuccess) return e;
  return launch(sort_small_kernel, 1, kSmallThreads, kSmallSmem, st, p);
}

// One LSD pass: 8-bit digits for the depth sort, 4 or 6 bits for the split by view.  The grid
// is at most one CTA per 2,048 items.  Up to kSortNoScan CTAs (32,768 items) every downsweep
// CTA reads the counts of all of them instead of a scan kernel's offsets: two launches instead
// of three; the 720p frame's 500,000 pairs (245 CTAs) are past the point where that reading
// costs more than the launch.
template <int BITS, int MODE>
static cudaError_t sort_pass(const SortPass &p, cudaStream_t st) {
  launch(sort_upsweep<BITS, MODE == kSortFirst>, p.G, kSortThreads, 0, st, p);
  if (p.G > kSortNoScan) launch(hist_scan_kernel, 1 << BITS, 256, 0, st, p.hist, p.G, p.digit_total);
  launch(sort_downsweep<BITS, MODE>, p.G, kSortThreads, 0, st, p);
  return cudaGetLastError();
}

int sort_blocks(uint64_t items, int grid) {
  const uint64_t need = (items + kSortTile - 1) / kSortTile;  // CTAs with work
  return need < uint64_t(grid) ? (need ? int(need) : 1) : grid;
}

cudaError_t launch_sort_pass(SortPass p, cudaStream_t st) {
  p.G = sort_blocks(p.count_max, p.G);
  if (p.row_info) return sort_pass<8, kSortFirst>(p, st);
  if (p.row_rect) return sort_pass<8, kSortLast>(p, st);
  if (!p.index_out) return sort_pass<8, kSortPlain>(p, st);
  return p.n_views <= 16 ? sort_pass<4, kSortSplit>(p, st) : sort_pass<6, kSortSplit>(p, st);
}

}  // namespace raygs
