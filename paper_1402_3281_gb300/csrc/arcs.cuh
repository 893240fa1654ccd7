// arcs.cuh -- streaming the arcs of a level in storage order, evenly split
// over the grid whatever the degrees are.
#pragma once
#include "common.cuh"

namespace sclap {

// The arcs are cut into tiles of AT_ARCS consecutive arcs; a CTA walks a
// contiguous range of arcs tile by tile.  Per tile it stages the row ends of
// the next AT_V nodes in shared memory, so an arc finds its source node by a
// search in shared memory; a thread holds AT_PER arcs, read as 16-byte words
// where the arrays allow it, so that many arcs and the gathers that depend on
// them are in flight.  A hub's row is simply many tiles.  (Before, a warp
// held 32 rows and took their arcs 32 at a time: one gather in flight per
// lane, and a hub's row was one warp's serial job.)
constexpr int AT_NT = 256;                 // threads per CTA
constexpr int AT_V = AT_NT;                // nodes staged per tile, one per thread
constexpr int AT_PER = 8;                  // arcs per thread and tile
constexpr int AT_ARCS = AT_NT * AT_PER;

// One thread's arcs of a tile: heads, weights, source nodes (-1: no arc).
struct ArcTile {
  int32_t c[AT_PER], w[AT_PER];
  int32_t v[AT_PER];
};

__device__ __forceinline__ bool arcs_aligned(const int32_t* col, const int32_t* ew) {
  return ((reinterpret_cast<uintptr_t>(col) | reinterpret_cast<uintptr_t>(ew)) & 15) == 0;
}

// Calls f(tile) for every tile of the arcs [lo, hi); all threads of the CTA
// call it equally often.  row_ptr is non-decreasing over [v0, v1] with
// row_ptr[v0] <= lo and hi <= row_ptr[v1] (v0 < v1); M is the length of col
// and ew (a 16-byte word reaching past it is read entry by entry); sh_end is
// AT_V words of shared memory.
template <class F>
__device__ __forceinline__ void for_arc_tiles(const int64_t* __restrict__ row_ptr, int64_t v0,
                                              int64_t v1, int64_t lo, int64_t hi,
                                              const int32_t* __restrict__ col,
                                              const int32_t* __restrict__ ew, int64_t M,
                                              int32_t* sh_end, F f) {
  if (lo >= hi) return;
  const int tid = threadIdx.x;
  const bool vec = arcs_aligned(col, ew);
  int64_t v = v0, b = v1 - 1;              // last node whose row starts at or before lo
  while (v < b) {
    const int64_t mid = (v + b + 1) >> 1;
    if (row_ptr[mid] <= lo) v = mid;
    else b = mid - 1;
  }
  while (lo < hi) {
    const int64_t u = v + tid + 1;
    int32_t end = AT_ARCS + 1;             // nodes past the range: no arc of the tile
    if (u <= v1) end = (int32_t)min64(row_ptr[u] - lo, AT_ARCS + 1);
    __syncthreads();                       // the previous tile's searches are done
    sh_end[tid] = end;
    __syncthreads();
    const int head = (int)(lo & 3);        // the tile's words start on 16-byte boundaries
    const int32_t span = (int32_t)min64(min64(AT_ARCS - head, hi - lo),
                                        max64(sh_end[AT_V - 1], 0));
    const int32_t x0 = tid * AT_PER - head;   // this thread's first arc, from lo
    const int64_t e0 = lo + x0;
    ArcTile t;
#pragma unroll
    for (int i = 0; i < AT_PER; ++i) {
      t.c[i] = 0;
      t.w[i] = ew ? 0 : 1;
      t.v[i] = -1;
    }
    if (x0 < span) {
      if (vec && e0 + AT_PER <= M) {
#pragma unroll
        for (int g = 0; g < AT_PER; g += 4) {
          const int4 c = *reinterpret_cast<const int4*>(col + e0 + g);
          t.c[g] = c.x; t.c[g + 1] = c.y; t.c[g + 2] = c.z; t.c[g + 3] = c.w;
          if (ew) {
            const int4 w = *reinterpret_cast<const int4*>(ew + e0 + g);
            t.w[g] = w.x; t.w[g + 1] = w.y; t.w[g + 2] = w.z; t.w[g + 3] = w.w;
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < AT_PER; ++i)
          if (x0 + i >= 0 && x0 + i < span) {
            t.c[i] = col[e0 + i];
            if (ew) t.w[i] = ew[e0 + i];
          }
      }
      // first staged node whose row ends after the first arc, then forward
      const int32_t xs = x0 > 0 ? x0 : 0;
      int j = 0, k = AT_V - 1;
      while (j < k) {
        const int mid = (j + k) >> 1;
        if (sh_end[mid] > xs) k = mid;
        else j = mid + 1;
      }
      int32_t ej = sh_end[j];
#pragma unroll
      for (int i = 0; i < AT_PER; ++i) {
        const int32_t x = x0 + i;
        if (x >= 0 && x < span) {
          while (ej <= x) ej = sh_end[++j];   // x < span <= sh_end[AT_V - 1]
          t.v[i] = (int32_t)v + j;
        }
      }
    }
    f(t);
    // the node that holds the next arc (the staged rows ending at or before it are done)
    int j = 0, k = AT_V;
    while (j < k) {
      const int mid = (j + k) >> 1;
      if (sh_end[mid] > span) k = mid;
      else j = mid + 1;
    }
    v += j;
    lo += span;
  }
}

// Arc range of this CTA: an even share of [0, M), whole tiles.
__device__ __forceinline__ void arc_share(int64_t M, int64_t* lo, int64_t* hi) {
  const int64_t per = ((M + gridDim.x - 1) / gridDim.x + AT_ARCS - 1) / AT_ARCS * AT_ARCS;
  *lo = min64((int64_t)blockIdx.x * per, M);
  *hi = min64(*lo + per, M);
}
// One wave of resident CTAs: the shares are even, so a second, partial wave
// would only add a tail.
constexpr int AT_CTAS = 6;                 // resident CTAs per SM (launch bounds)
inline unsigned arc_grid(int64_t M) {
  return grid_for(M, AT_ARCS, (int64_t)num_sms() * AT_CTAS);
}

// Last slot s with off[s] <= x (off non-decreasing, off[0] = 0): the slot of
// an arc, or of a node, that exists (empty slots before it are passed over).
__device__ __forceinline__ int32_t slot_of(const int64_t* __restrict__ off, int32_t nslots,
                                           int64_t x) {
  int32_t lo = 0, hi = nslots - 1;
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (off[mid] <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Sum over the CTA (valid in thread 0); sh holds one word per warp.
__device__ __forceinline__ unsigned long long cta_sum(unsigned long long x,
                                                      unsigned long long* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  __syncthreads();
  if (lane == 0) sh[wid] = x;
  __syncthreads();
  unsigned long long t = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
  return t;
}

}  // namespace sclap
