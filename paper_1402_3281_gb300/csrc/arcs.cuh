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
constexpr int AT_V = AT_NT;                // rows staged per tile by one row per thread
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

// Last row of [v, v1) that starts at or before lo, by a search in doubling
// steps from v (row_ptr[v] <= lo < row_ptr[v1]).
static __device__ __noinline__ int32_t row_after_gap(const int64_t* row_ptr, int32_t v, int32_t v1,
                                                     int64_t lo) {
  int32_t step = AT_V;
  while (step < v1 - v && row_ptr[v + step] <= lo) {
    v += step;
    step = step < (1 << 29) ? 2 * step : step;
  }
  for (; step > 0; step /= 2)              // the row is less than step rows on
    if (step < v1 - v && row_ptr[v + step] <= lo) v += step;
  return v;
}

// Walks the entries [lo, hi) of rows laid out back to back (arcs of nodes,
// slots of table regions) tile by tile: calls f(lo, span, v) for the tile of
// the entries [lo, lo + span), whose rows are v .. v + R * AT_V - 1 with ends
// sh_end[j] (relative to lo; R * AT_V rows, R per thread).  All threads of the CTA call it equally often.
// row_ptr is non-decreasing over [v0, v1] with row_ptr[v0] <= lo and
// hi <= row_ptr[v1] (v0 < v1); sh_end is R * AT_V words of shared memory.  A tile
// never reaches past the AT_ARCS entries from lo rounded down to 4.
//
// A run of rows without entries is passed over by a search in doubling steps:
// staging it 256 rows at a time was a serial job of the one CTA that met it
// while the rest of the grid was done (a path of 1 M nodes with ten million
// isolated nodes in the middle: a cut 74 -> 0.18 ms, a contraction 281 -> 0.78).
template <int R = 1, class F>
__device__ __forceinline__ void for_tiles(const int64_t* __restrict__ row_ptr, int64_t v0,
                                          int64_t v1, int64_t lo, int64_t hi, int32_t* sh_end,
                                          F f) {
  if (lo >= hi) return;
  const int tid = threadIdx.x;
  // (rows are numbered below 2^31)
  const int32_t vend = (int32_t)v1;
  int32_t v = (int32_t)v0;                 // last row that starts at or before lo
  for (int32_t b = vend - 1; v < b;) {
    const int32_t mid = v + (b - v + 1) / 2;
    if (row_ptr[mid] <= lo) v = mid;
    else b = mid - 1;
  }
  while (lo < hi) {
    int32_t end[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int32_t j = r * AT_V + tid;
      end[r] = AT_ARCS + 1;                // rows past the range: no entry of the tile
      if (j < vend - v) end[r] = (int32_t)max64(min64(row_ptr[v + j + 1] - lo, AT_ARCS + 1), 0);
    }
    __syncthreads();                       // the previous tile's searches are done
#pragma unroll
    for (int r = 0; r < R; ++r) sh_end[r * AT_V + tid] = end[r];
    __syncthreads();
    if (sh_end[R * AT_V - 1] == 0) {           // none of the staged rows reaches past lo
      v = row_after_gap(row_ptr, v + R * AT_V, vend, lo);
      continue;
    }
    const int32_t span = (int32_t)min64(min64(AT_ARCS - (int)(lo & 3), hi - lo), sh_end[R * AT_V - 1]);
    f(lo, span, (int64_t)v);
    // the row that holds the next entry (the staged rows ending at or before it are done)
    int j = 0, k = R * AT_V;
    while (j < k) {
      const int mid = (j + k) >> 1;
      if (sh_end[mid] > span) k = mid;
      else j = mid + 1;
    }
    v += j;
    lo += span;
  }
}

// Rows (j: from the tile's first; -1: no entry) of this thread's AT_PER
// consecutive entries, which start at x0 from the tile's first: a search for
// the first, then forward.
template <int R = 1>
__device__ __forceinline__ void tile_rows(const int32_t* sh_end, int32_t x0, int32_t span,
                                          int32_t (&row)[AT_PER]) {
  const int32_t xs = x0 > 0 ? x0 : 0;
  int j = 0, k = R * AT_V - 1;
  while (j < k) {
    const int mid = (j + k) >> 1;
    if (sh_end[mid] > xs) k = mid;
    else j = mid + 1;
  }
  int32_t ej = sh_end[j];
#pragma unroll
  for (int i = 0; i < AT_PER; ++i) {
    const int32_t x = x0 + i;
    row[i] = -1;
    if (x >= 0 && x < span) {
      while (ej <= x) ej = sh_end[++j];    // x < span <= the last sh_end
      row[i] = j;
    }
  }
}

// Calls f(tile, v, span) for every tile of the arcs [lo, hi) (see for_tiles; v:
// the tile's first staged node).  M is the length of col and ew: a 16-byte word
// reaching past it is read entry by entry.
template <int R = 1, class F>
__device__ __forceinline__ void for_arc_tiles(const int64_t* __restrict__ row_ptr, int64_t v0,
                                              int64_t v1, int64_t lo, int64_t hi,
                                              const int32_t* __restrict__ col,
                                              const int32_t* __restrict__ ew, int64_t M,
                                              int32_t* sh_end, F f) {
  const bool vec = arcs_aligned(col, ew);
  for_tiles<R>(row_ptr, v0, v1, lo, hi, sh_end, [&](int64_t lo, int32_t span, int64_t v) {
    // the tile's words start on 16-byte boundaries
    const int32_t x0 = (int32_t)threadIdx.x * AT_PER - (int32_t)(lo & 3);
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
      tile_rows<R>(sh_end, x0, span, t.v);
#pragma unroll
      for (int i = 0; i < AT_PER; ++i)
        if (t.v[i] >= 0) t.v[i] += (int32_t)v;
    }
    f(t, v, span);
  });
}

// Arc range of this CTA: an even share of [0, M), whole tiles, or on levels
// with fewer arcs than that (arc_grid) a part of one.
__device__ __forceinline__ void arc_share(int64_t M, int64_t* lo, int64_t* hi) {
  int64_t per = (M + gridDim.x - 1) / gridDim.x;
  const int64_t unit = per < AT_ARCS ? 4 : AT_ARCS;
  per = (per + unit - 1) / unit * unit;
  *lo = min64((int64_t)blockIdx.x * per, M);
  *hi = min64(*lo + per, M);
}
// One wave of resident CTAs: the shares are even, so a second, partial wave
// would only add a tail.  A CTA per tile of arcs or per eight staged blocks of
// rows, whichever are more: with far fewer arcs than rows the steps over the
// rows are the work (10 M nodes, 20,000 arcs: a cut 6.7 -> 0.23 ms, a
// contraction 24.7 -> 0.9).
constexpr int AT_CTAS = 6;                 // resident CTAs per SM (launch bounds)
inline unsigned arc_grid(int64_t M, int64_t rows, int ctas = AT_CTAS) {
  return grid_for(M > rows ? M : rows, AT_ARCS, (int64_t)num_sms() * ctas);
}

// Rows staged per thread where rows are short: one row per thread holds fewer
// entries than a tile when rows average below AT_ARCS / AT_V, and then the
// steps over the rows (two barriers each) are the work.  Staging four:
// contraction of a mesh of 4 M nodes and degree 4 1.39 -> 1.11 ms, of R-MAT
// 2^22 nodes and 8.3 M arcs 2.61 -> 1.44, of 10 M nodes and 2 M arcs 1.56 ->
// 0.98; cuts of the three 0.21 -> 0.17, 0.27 -> 0.18 and 0.47 -> 0.25 ms.  At
// degree 6 5 to 7 % faster, at 8 and above no different.
constexpr int SHORT_ROWS = 4;
inline bool rows_short(int64_t entries, int64_t rows) { return entries < AT_ARCS / AT_V * rows; }

// Exclusive prefix of x over the CTA's threads (AT_NT); sh holds AT_NT / 32
// words, all threads call.
__device__ __forceinline__ int32_t cta_excl(int32_t x, int32_t* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t inc = x;
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  __syncthreads();
  if (lane == 31) sh[wid] = inc;
  __syncthreads();
  int32_t before = 0;
  for (int w = 0; w < wid; ++w) before += sh[w];
  return before + inc - x;
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
