// Stable expansion of intervals into per-bin lists, shared by the two levels of the binning
// (pairs -> tile rows of their view, support rows -> tile columns of their tile row).
//
// Items come in depth order; each covers the bins [first, first + len).  A warp takes 32
// items at a time.  Every item toggles its lane's bit at its first bin and past its last
// one; the running XOR over the bins is then, per bin, the mask of the lanes that cover it,
// so that the rank of (item, bin) is the bin's cursor plus the mask's bits below the item's
// lane.  Two shared-memory atomics per item, whatever it covers, and no barrier beyond the
// warp.  The instances of the 32 items are then taken 32 at a time, one per lane.
//
// Lane l owns the bins [l J, (l + 1) J), J odd (no bank conflicts), their cursors in registers.  The counts
// work for a run-time number of bins per lane too (J = 0).
#pragma once

#include "raygs_internal.cuh"

namespace raygs {

// bins per lane so that 32 nj > bins (the toggle past the last bin has a slot too)
__host__ __device__ inline int bins_per_lane(int bins) { return (bins / 32 + 1) | 1; }

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// Block-wide exclusive scan (blockDim.x multiple of 32, <= 1024).  Returns the exclusive
// prefix; *total receives the block total.  Uses `ws` (>= 33 words of shared memory).
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t *ws, uint32_t *total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t inc = warp_incl_scan(x);
  if (lane == 31) ws[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t v = lane < nw ? ws[lane] : 0u;
    uint32_t vi = warp_incl_scan(v);
    if (lane < nw) ws[lane] = vi - v;
    if (lane == nw - 1) ws[32] = vi;
  }
  __syncthreads();
  uint32_t r = inc - x + ws[warp];
  *total = ws[32];
  __syncthreads();
  return r;
}

// Items per bin from a difference array (+1 at an item's first bin, -1 past its last one);
// clears the array.  One warp; __syncwarp() before and after.
template <int J>
__device__ __forceinline__ void bins_counts(uint32_t *diff, uint32_t *cnt, int nj_dyn) {
  const int nj = J ? J : nj_dyn, b0 = (threadIdx.x & 31) * nj;
  uint32_t s = 0;
#pragma unroll(J ? J : 1)
  for (int j = 0; j < nj; ++j) s += diff[b0 + j];
  uint32_t run = warp_incl_scan(s) - s;
#pragma unroll(J ? J : 1)
  for (int j = 0; j < nj; ++j) {
    run += diff[b0 + j];
    diff[b0 + j] = 0u;
    cnt[b0 + j] = run;
  }
}

// Masks of 32 items from their toggles: mc[b] = (lanes covering b, cursor of b before these
// items); the cursors advance past them and the toggles are cleared.
template <int J>
__device__ __forceinline__ void bins_masks(uint32_t *tog, uint2 *mc, uint32_t (&cur)[J]) {
  const int lane = threadIdx.x & 31, b0 = lane * J;
  uint32_t loc[J], x = 0;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    x ^= tog[b0 + j];
    tog[b0 + j] = 0u;
    loc[j] = x;
  }
  uint32_t s = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
    if (lane >= o) s ^= y;
  }
  const uint32_t carry = s ^ x;  // toggles of the lower lanes' bins
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const uint32_t m = loc[j] ^ carry;
    mc[b0 + j] = make_uint2(m, cur[j]);
    cur[j] += __popc(m);
  }
  __syncwarp();
}

// Owner of instance i = base + lane among the items whose instances start at `start` (in
// item order): the ordinal of the last non-empty item that starts at or before i.  `seen`
// carries the items that started before base (0 at first).
__device__ __forceinline__ int instance_owner(uint32_t start, bool nonempty, uint32_t base, uint32_t &seen) {
  const int lane = threadIdx.x & 31;
  const uint32_t rel = start - base;
  const uint32_t w = __reduce_or_sync(0xffffffffu, nonempty && rel < 32u ? 1u << rel : 0u);
  const int k = int(seen + __popc(w & (0xFFFFFFFFu >> (31 - lane)))) - 1;
  seen += __popc(w);
  return k;
}

}  // namespace raygs
