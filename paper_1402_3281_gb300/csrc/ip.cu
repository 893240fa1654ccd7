// ip.cu -- initial partitioning of the coarsest graphs, cut, projection.
//
// The paper partitions the coarsest graph with KaHIP's recursive bisection,
// which it does not specify.  Here every graph gets `trials` independent
// trials, all graphs' trials forming one batch: greedy graph growing (one CTA
// per trial: block j starts at a hashed seed and absorbs the unassigned
// nodes connected to it, in node-id order, while it stays <= ceil(c(V)/k)),
// water-filling of the leftovers, then LP local search (the lp.cu kernels on
// the whole trial batch).  The best trial by (overload, cut, trial) is kept.
#include <algorithm>

#include "arcs.cuh"

namespace sclap {
namespace {

// CTA sizes of the greedy-growing kernel: 128 threads when a batch has many
// trials (more trials in flight), 512 when it has few (wider steps).
constexpr int GNT_MANY = 128, GNT_FEW = 1024;
constexpr int GPER = 8;   // consecutive nodes per thread in the greedy-growing scans
// arcs per thread per pass in the greedy-growing accumulation (more in the
// wide CTAs, which have the registers and run on few trials)
template <int GNT> struct Garc { static constexpr int value = GNT >= 512 ? 8 : 4; };

// All copies of a graph segment from one read of it: a thread holds RP_PER
// arcs and stores them once per copy, so a graph with 16 trials moves 17
// streams instead of 31 and its neighbours are renumbered once.  Bound by the
// stores; four arcs in flight per thread cover the rank gather.  blockIdx.z
// shares out the copies where a segment alone has too few tiles for the chip.
// Two passes (copy, then copies of the copy) -> this: 16 copies of an R-MAT
// graph of 2^22 nodes 2.35 -> 1.1 ms, of 512 small graphs 1.45 -> 0.72 ms.
// (5 TB/s of stores at 2^22 nodes; 54 GB of copies of a 2^24-node graph take
// 33 ms either way, 1.6 TB/s: streaming stores, a copy per CTA row, longer
// tiles and renumbering in a pass of its own gave 28 to 36 ms.)
constexpr int RP_NT = 256, RP_PER = 4;
__global__ void __launch_bounds__(RP_NT) k_replicate(const CopyTask* __restrict__ tasks,
                                                     int64_t* __restrict__ row_ptr,
                                                     int32_t* __restrict__ col,
                                                     int32_t* __restrict__ ew,
                                                     int32_t* __restrict__ nw) {
  const CopyTask t = tasks[blockIdx.y];
  const int64_t tile = RP_NT * RP_PER, stride = (int64_t)gridDim.x * tile;
  const int c0 = (int)blockIdx.z, cs = (int)gridDim.z;
  for (int64_t b = (int64_t)blockIdx.x * tile; b < t.n; b += stride) {
    int64_t d[RP_PER], r[RP_PER];
    int32_t w[RP_PER];
#pragma unroll
    for (int i = 0; i < RP_PER; ++i) {
      const int64_t v = b + i * RP_NT + threadIdx.x;
      const bool in = v < t.n;
      d[i] = in ? v : -1;
      r[i] = in ? t.row_ptr[t.src_n0 + v] - t.src_a0 : 0;
      w[i] = in && nw ? wat(t.nw, t.src_n0 + v) : 0;
      if (in && t.rank) {
        const int64_t x = t.rank[t.src_n0 + v];
        d[i] = t.rank[t.src_n0 + v + 1] == x ? -1 : x - t.rbase;   // isolated: dropped
      }
    }
    for (int64_t c = c0; c < t.copies; c += cs) {
      const int64_t n0 = t.dst_n0 + c * t.nd, a0 = t.dst_a0 + c * t.m;
#pragma unroll
      for (int i = 0; i < RP_PER; ++i)
        if (d[i] >= 0) {
          row_ptr[n0 + d[i]] = a0 + r[i];
          if (nw) nw[n0 + d[i]] = w[i];
        }
    }
  }
  for (int64_t b = (int64_t)blockIdx.x * tile; b < t.m; b += stride) {
    int64_t u[RP_PER];
    int32_t w[RP_PER];
#pragma unroll
    for (int i = 0; i < RP_PER; ++i) {
      const int64_t e = b + i * RP_NT + threadIdx.x;
      u[i] = e < t.m ? (int64_t)t.col[t.src_a0 + e] : t.src_n0;
      w[i] = e < t.m && ew ? wat(t.ew, t.src_a0 + e) : 0;
    }
#pragma unroll
    for (int i = 0; i < RP_PER; ++i)
      u[i] = t.rank ? t.rank[u[i]] - t.rbase : u[i] - t.src_n0;   // (unchecked input: any int32)
    for (int64_t c = c0; c < t.copies; c += cs) {
      const int64_t n0 = t.dst_n0 + c * t.nd, a0 = t.dst_a0 + c * t.m + b + threadIdx.x;
#pragma unroll
      for (int i = 0; i < RP_PER; ++i)
        if (b + i * RP_NT + threadIdx.x < t.m) {
          col[a0 + i * RP_NT] = (int32_t)(u[i] + n0);
          if (ew) ew[a0 + i * RP_NT] = w[i];
        }
    }
  }
}

__global__ void k_set_i64(int64_t* p, int64_t v) { *p = v; }

// Block-wide inclusive scan of an int64 (all GNT threads call it).
template <int GNT>
__device__ int64_t block_incl_scan(int64_t x, int64_t* sh, int64_t* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, (long long)x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int64_t v = lane < GNT / 32 ? sh[lane] : 0;
    int64_t vi = v;
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, (long long)vi, o);
      if (lane >= o) vi += y;
    }
    if (lane < GNT / 32) sh[lane] = vi - v;
    if (lane == 31) sh[32] = vi;
  }
  __syncthreads();
  x += sh[wid];
  *total = sh[32];
  __syncthreads();
  return x;
}

template <int GNT>
__device__ int64_t block_sum(int64_t x, int64_t* sh) {
  int64_t tot;
  block_incl_scan<GNT>(x, sh, &tot);
  return tot;
}

// Bitmaps of greedy growing, one bit per node of a trial, each trial in words
// of its own: assigned nodes, and nodes seen (assigned, or reached by the
// block that is growing).  Which nodes a step may absorb depends only on
// whether a node is connected to the block, not on how strongly, so a reached
// bit is all an arc has to leave behind.
__host__ __device__ __forceinline__ int64_t ggg_word0(int64_t noff, int64_t slot) {
  return (noff >> 5) + slot;               // disjoint: every trial may round up by one word
}
__host__ __device__ __forceinline__ int64_t ggg_words(int64_t n) { return (n + 31) >> 5; }

// One CTA per trial.  The chain of small steps of a trial is what bounds it,
// so what a step waits for is kept close: the bitmaps lie in shared memory up
// to GGG_SHW words (32,768 nodes), where the connection sums were random
// global atomics.  Measured: all trials of the 512-graph batch 2.53 -> 1.42
// ms, of one 2^22-node mesh (k = 64) 1.93 -> 1.37 ms.
constexpr int GGG_SHW = 1024;
template <int GNT>
__global__ void __launch_bounds__(GNT) k_ggg(GGGArgs a) {
  constexpr int GARC = Garc<GNT>::value;
  __shared__ int64_t sh[33];
  __shared__ uint64_t shh[GNT / 32];
  __shared__ int32_t shv[GNT / 32];
  __shared__ int64_t Wj_sh;
  __shared__ unsigned long long accw_sh;
  __shared__ int32_t nstep_sh, seed_sh, nfront_sh;
  // a chunk of step nodes: one past the last arc offset of each, and what
  // turns an arc offset into an arc of the level
  __shared__ int64_t st_in[GNT], st_off[GNT];
  __shared__ int32_t next_sh;
  __shared__ uint32_t sh_asg[GGG_SHW], sh_seen[GGG_SHW];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  // trials are taken from a queue ordered by size, largest first, so the
  // long trials of the batch start first and on different CTAs
  for (;;) {
    if (tid == 0) next_sh = atomicAdd(a.next, 1);
    __syncthreads();
    const int32_t qi = next_sh;
    __syncthreads();
    if (qi >= a.nslots) break;
    const int32_t s = a.order[qi];
    const int64_t base = a.noff[s], n = a.noff[s + 1] - base;
    const int32_t k = a.nlab[s];
    const int64_t bo = a.boff[s], avg = a.avg[s];
    const uint64_t tkey = a.tkey[s];
    const int32_t lvl = a.level[s];
    const int64_t nwords = ggg_words(n), nbytes = (n + GPER - 1) / GPER;
    const bool in_sh = nwords <= GGG_SHW;
    uint32_t* asg = in_sh ? sh_asg : a.asg + ggg_word0(base, s);
    uint32_t* seen = in_sh ? sh_seen : a.seen + ggg_word0(base, s);
    auto bit_of = [](const uint32_t* m, int64_t v) { return (m[v >> 5] >> (v & 31)) & 1u; };
    for (int64_t w = tid; w < nwords; w += GNT) asg[w] = 0;
    for (int32_t b = tid; b < k; b += GNT) a.W[bo + b] = 0;
    __syncthreads();
    for (int32_t j = 0; j < k; ++j) {
      // seed: unassigned non-isolated node with the smallest hash (the row is
      // looked at only for a node that would be taken)
      const uint64_t skey = hkey(tkey, PH_GGG, (uint64_t)lvl, (uint64_t)j);
      uint64_t bh = ~0ull;
      int32_t bv = -1;
      for (int64_t v = tid; v < n; v += GNT) {
        if (bit_of(asg, v)) continue;
        const uint64_t h = mix64(skey ^ (uint64_t)v);
        if ((bv < 0 || h < bh) && a.row_ptr[base + v + 1] != a.row_ptr[base + v]) {
          bh = h;
          bv = (int32_t)v;
        }
      }
      // (nothing is reached yet)
      for (int64_t w = tid; w < nwords; w += GNT) seen[w] = asg[w];
      for (int o = 16; o > 0; o >>= 1) {
        uint64_t oh = __shfl_xor_sync(0xffffffffu, (unsigned long long)bh, o);
        int32_t ov = __shfl_xor_sync(0xffffffffu, bv, o);
        if (ov >= 0 && (bv < 0 || oh < bh || (oh == bh && ov < bv))) { bh = oh; bv = ov; }
      }
      if (lane == 0) { shh[wid] = bh; shv[wid] = bv; }
      __syncthreads();
      // step nodes and newly reached nodes: two scratch lists that swap roles
      int32_t* stp = a.step + base;
      int32_t* frt = a.front + base;
      if (tid == 0) {
        uint64_t h = ~0ull;
        int32_t v = -1;
        for (int w = 0; w < GNT / 32; ++w)
          if (shv[w] >= 0 && (v < 0 || shh[w] < h || (shh[w] == h && shv[w] < v))) {
            h = shh[w]; v = shv[w];
          }
        seed_sh = v;
        if (v >= 0) {
          a.label[base + v] = (int32_t)(bo + j);
          asg[v >> 5] |= 1u << (v & 31);
          seen[v >> 5] |= 1u << (v & 31);
          stp[0] = (int32_t)(base + v);
          nstep_sh = 1;
          nfront_sh = 0;
          Wj_sh = a.nw[base + v];
          accw_sh = 0;
        }
      }
      __syncthreads();
      if (seed_sh < 0) break;
      // while every step has absorbed all its candidates, the candidates of
      // the next step are exactly the nodes first reached by this one, listed
      // as they are reached; the first step whose candidates do not all fit
      // switches the block to the ordered scan over the reached nodes
      bool ordered = false;
      while (true) {
        // the arcs of up to GNT step nodes at a time are spread over all
        // threads (a hub in the step does not hold back one warp)
        const int32_t nstep = nstep_sh;
        const int64_t Wj = Wj_sh;
        if (Wj >= avg) break;
        unsigned long long fw = 0;   // weight of the nodes this thread listed
        for (int32_t q0 = 0; q0 < nstep; q0 += GNT) {
          const int32_t q = q0 + tid;
          int64_t rs = 0, d = 0;
          if (q < nstep) {
            const int32_t u = stp[q];
            rs = a.row_ptr[u];
            d = a.row_ptr[u + 1] - rs;
          }
          int64_t tot;
          const int64_t incl = block_incl_scan<GNT>(d, sh, &tot);
          st_in[tid] = incl;
          st_off[tid] = rs - (incl - d);
          __syncthreads();
          const int cnt = min(GNT, nstep - q0);
          // up to GARC consecutive arcs per thread per pass: one owner search
          // for all of them, and their loads overlap (fewer while that keeps
          // more threads busy: a small step is a chain of latencies)
          const int per = (int)min64(GARC, (tot + GNT - 1) / GNT);
          for (int64_t x0 = (int64_t)tid * per; x0 < tot; x0 += (int64_t)GNT * per) {
            // owner: the first step node whose arcs end after x0 (skips step
            // nodes without arcs), then forward
            int lo = 0, hi = cnt - 1;
            while (lo < hi) {
              const int mid = (lo + hi) >> 1;
              if (st_in[mid] > x0) hi = mid; else lo = mid + 1;
            }
            int32_t y[GARC];
#pragma unroll
            for (int u = 0; u < GARC; ++u) {
              const int64_t x = x0 + u;
              y[u] = -1;
              if (u >= per || x >= tot) continue;
              while (st_in[lo] <= x) ++lo;
              const int32_t g = a.col[st_off[lo] + x];
              y[u] = SCLAP_OK(g, a.N, a.err) ? (int32_t)(g - base) : -1;
            }
            uint32_t wd[GARC];
#pragma unroll
            for (int u = 0; u < GARC; ++u) wd[u] = y[u] >= 0 ? seen[y[u] >> 5] : ~0u;
#pragma unroll
            for (int u = 0; u < GARC; ++u) {
              const uint32_t bit = 1u << (y[u] & 31);
              if (wd[u] & bit) continue;           // (also y < 0)
              if (atomicOr(&seen[y[u] >> 5], bit) & bit) continue;
              if (!ordered) {                      // reached for the first time
                frt[atomicAdd(&nfront_sh, 1)] = (int32_t)(base + y[u]);
                fw += (unsigned long long)a.nw[base + y[u]];
              }
            }
          }
          __syncthreads();
        }
        if (!ordered) {
          for (int o = 16; o > 0; o >>= 1) fw += __shfl_xor_sync(0xffffffffu, fw, o);
          if (lane == 0 && fw) atomicAdd(&accw_sh, fw);
          __syncthreads();
          const int64_t fsum = (int64_t)accw_sh;
          const int32_t nf = nfront_sh;
          if (Wj + fsum <= avg) {
            // all of them fit: they are the next step, in any order
            for (int32_t q = tid; q < nf; q += GNT) {
              const int32_t g = frt[q];
              const int64_t v = g - base;
              a.label[g] = (int32_t)(bo + j);
              atomicOr(&asg[v >> 5], 1u << (v & 31));
            }
            int32_t* t = stp; stp = frt; frt = t;
            __syncthreads();
            if (tid == 0) {
              nstep_sh = nf;
              nfront_sh = 0;
              accw_sh = 0;
              Wj_sh = Wj + fsum;
            }
            __syncthreads();
            if (nf == 0) break;
            continue;
          }
          ordered = true;
          __syncthreads();
          if (tid == 0) { nfront_sh = 0; accw_sh = 0; }
          __syncthreads();
        }
        // reached unassigned nodes in id order, longest prefix that fits: a
        // thread takes GPER consecutive nodes (a byte of the bitmaps) per
        // pass, a block scan gives its offset; the list's order is free
        int64_t carry_w = 0;
        unsigned long long acc_w = 0;
        for (int64_t c0 = 0; c0 < nbytes; c0 += GNT) {
          const int64_t c = c0 + tid;
          uint32_t m = 0;
          if (c < nbytes)
            m = ((seen[c >> 2] & ~asg[c >> 2]) >> ((c & 3) * 8)) & 0xffu;
          int32_t wt[GPER];
          int64_t tsum = 0;
#pragma unroll
          for (int i = 0; i < GPER; ++i) {
            wt[i] = (m >> i) & 1u ? a.nw[base + c * GPER + i] : 0;
            tsum += wt[i];
          }
          int64_t tw;
          int64_t run = Wj + carry_w + block_incl_scan<GNT>(tsum, sh, &tw) - tsum;
          uint32_t adm = 0;
#pragma unroll
          for (int i = 0; i < GPER; ++i) {
            run += wt[i];
            if (((m >> i) & 1u) && run <= avg) {
              adm |= 1u << i;
              acc_w += (unsigned long long)wt[i];
            }
          }
          if (adm) {
            int32_t pos = atomicAdd(&nfront_sh, __popc(adm));
#pragma unroll
            for (int i = 0; i < GPER; ++i)
              if ((adm >> i) & 1u) stp[pos++] = (int32_t)(base + c * GPER + i);
          }
          carry_w += tw;
          if (Wj + carry_w > avg) break;   // no later candidate can fit
        }
        if (acc_w) atomicAdd(&accw_sh, acc_w);
        __syncthreads();
        const int32_t ns2 = nfront_sh;
        for (int32_t q = tid; q < ns2; q += GNT) {
          const int32_t g = stp[q];
          const int64_t v = g - base;
          a.label[g] = (int32_t)(bo + j);
          atomicOr(&asg[v >> 5], 1u << (v & 31));
        }
        __syncthreads();
        if (tid == 0) {
          nstep_sh = ns2;
          nfront_sh = 0;
          Wj_sh = Wj + (int64_t)accw_sh;
          accw_sh = 0;
        }
        __syncthreads();
        if (ns2 == 0) break;
      }
      if (tid == 0) a.W[bo + j] = (wgt_t)Wj_sh;
      __syncthreads();
    }
    // water-filling of the nodes left unassigned
    int64_t r = 0;
    for (int64_t v = tid; v < n; v += GNT)
      if (!bit_of(asg, v)) r += a.nw[base + v];
    const int64_t R = block_sum<GNT>(r, sh);
    if (R > 0) {
      if (tid == 0) {
        int64_t lo = a.W[bo], hi = a.W[bo];
        for (int32_t b = 1; b < k; ++b) {
          lo = min64(lo, (int64_t)a.W[bo + b]);
          hi = max64(hi, (int64_t)a.W[bo + b]);
        }
        hi += R;
        while (lo < hi) {
          const int64_t mid = lo + (hi - lo) / 2;
          int64_t f = 0;
          for (int32_t b = 0; b < k; ++b) f += max64(0, mid - (int64_t)a.W[bo + b]);
          if (f >= R) hi = mid; else lo = mid + 1;
        }
        const int64_t L = lo;
        for (int32_t j = 0; j < k; ++j) {       // insertion sort by (W, id)
          int32_t b = j;
          int32_t p = j;
          while (p > 0) {
            const int32_t q = a.wforder[bo + p - 1];
            if (a.W[bo + q] > a.W[bo + b] || (a.W[bo + q] == a.W[bo + b] && q > b)) {
              a.wforder[bo + p] = q;
              --p;
            } else {
              break;
            }
          }
          a.wforder[bo + p] = b;
        }
        int64_t acc = 0;
        for (int32_t j = 0; j < k; ++j) {
          a.wfA[bo + j] = acc;
          acc += max64(0, L - (int64_t)a.W[bo + a.wforder[bo + j]]);
        }
      }
      __syncthreads();
      int64_t carry = 0;
      for (int64_t v0 = 0; v0 < n; v0 += GNT) {
        const int64_t v = v0 + tid;
        const bool left = v < n && !bit_of(asg, v);
        const int64_t wt = left ? a.nw[base + v] : 0;
        int64_t tw;
        const int64_t iw = block_incl_scan<GNT>(wt, sh, &tw);
        if (left) {
          const int64_t p = carry + iw - wt;
          int32_t lo = 0, hi = k - 1;               // last j with A[j] <= p
          while (lo < hi) {
            const int32_t mid = (lo + hi + 1) >> 1;
            if (a.wfA[bo + mid] <= p) lo = mid; else hi = mid - 1;
          }
          const int32_t b = a.wforder[bo + lo];
          a.label[base + v] = (int32_t)(bo + b);
          atomicAdd(&a.W[bo + b], (wgt_t)wt);
        }
        carry += tw;
      }
      __syncthreads();
    }
  }
}

// ------------------------------------------------------------------------
// Greedy growing of few, large trials: each trial is grown by a group of cpt
// CTAs of one cooperative launch (CTAs g * cpt .. g * cpt + cpt - 1 grow
// trial slot g), with the same rules as k_ggg.  The group shares the
// trial's step and front lists and a few counters in global memory and
// meets at a barrier of its own (bounded wait: a wait that runs out sets
// DERR_TIMEOUT and the group leaves; the labels are valid blocks from the
// start, k_first_blocks).  Each CTA owns a contiguous range of
// the trial's nodes for the scans (seed search, ordered candidates,
// water-filling); id-ordered prefixes over the whole trial are the CTAs'
// partial sums in rank order plus the CTA's own scan.  The step nodes'
// arcs are shared out by step node in chunks of GG_NT per CTA; a step node
// with more than GG_HEAVY arcs (known in advance: the step that builds the
// next step records whether it took one) is listed instead, and after a
// group barrier the listed rows are read by all CTAs of the group together.
// Every decision is a set or an id-ordered prefix, so the result equals
// k_ggg's.
struct GroupState {
  GridSync bar;
  int32_t nstep, nfront, nnext, seed;
  int64_t Wj, fsum, accw;
  // heavy step nodes (more than GG_HEAVY arcs): whether the current step
  // has any, whether the frontier / the ordered selection being built took
  // one, and the current step's list length
  int32_t step_heavy, front_heavy, next_heavy, nheavy;
};
constexpr int GG_NT = 512;
constexpr int64_t GG_HEAVY = 8 * GG_NT;

// The arc passes read and set one bit per arc: the seen bitmap (a bit per
// node and trial) stays in L2, where 64-bit connection sums (random atomics
// on arrays far larger than L2, before) did not, and an arc to a node
// already seen costs a read only.  What then bounds the pass is instruction
// issue, so a thread takes consecutive arcs and searches their source once.
// Measured, R-MAT 2^24 nodes (16 trials, 7.6 G arc visits): 101 -> 74 ms with
// the bitmaps, 43 ms with consecutive arcs; 2^22 nodes 14.1 -> 6.1 ms.
constexpr int GG_ARC = 8;                  // arcs per thread and pass

// Every node of the trials in its trial's first block, and empty blocks: a
// group whose wait runs out leaves nodes that it never reached, and what
// follows indexes block arrays by the labels until the host reads the error.
__global__ void __launch_bounds__(256) k_first_blocks(GGGArgs a) {
  const int32_t s = (int32_t)blockIdx.y;
  const int64_t base = a.noff[s], n = a.noff[s + 1] - base, bo = a.boff[s];
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    a.label[base + v] = (int32_t)bo;
  if (blockIdx.x == 0)
    for (int32_t b = threadIdx.x; b < a.nlab[s]; b += blockDim.x) a.W[bo + b] = 0;
}

__global__ void __launch_bounds__(GG_NT) k_ggg_group(GGGArgs a, int32_t cpt, GroupState* gst,
                                                     uint64_t* ph, int32_t* pv, int64_t* pw,
                                                     uint32_t lim) {
  __shared__ int64_t sh[33];
  __shared__ uint64_t shh[GG_NT / 32];
  __shared__ int32_t shv[GG_NT / 32];
  // a chunk of step nodes: one past the last arc offset of each (at most
  // GG_NT * GG_HEAVY), and what turns an arc offset into an arc
  __shared__ int32_t st_in[GG_NT];
  __shared__ int64_t st_off[GG_NT];
  __shared__ int64_t pre_sh, tot_sh;
  __shared__ int32_t seed_sh;
  // a bounded wait of an earlier launch ran out: the call is abandoned
  if (*(volatile int32_t*)a.err & DERR_TIMEOUT) return;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int32_t s = (int32_t)(blockIdx.x / cpt);
  const int r = (int)(blockIdx.x % cpt);
  GroupState* st = gst + s;
  uint64_t* gph = ph + (int64_t)s * cpt;
  int32_t* gpv = pv + (int64_t)s * cpt;
  int64_t* gpw = pw + (int64_t)s * cpt;
  const int64_t base = a.noff[s], n = a.noff[s + 1] - base;
  const int32_t k = a.nlab[s];
  const int64_t bo = a.boff[s], avg = a.avg[s];
  const uint64_t tkey = a.tkey[s];
  const int32_t lvl = a.level[s];
  // this CTA's node range, whole words of the bitmaps
  const int64_t nwords = ggg_words(n);
  const int64_t wr0 = nwords * r / cpt, wr1 = nwords * (r + 1) / cpt;
  const int64_t r0 = wr0 * 32, r1 = min64(wr1 * 32, n);
  uint32_t* asg = a.asg + ggg_word0(base, s);
  uint32_t* seen = a.seen + ggg_word0(base, s);
  auto bit_of = [](const uint32_t* m, int64_t v) { return (m[v >> 5] >> (v & 31)) & 1u; };
  const int64_t qstride = (int64_t)GG_NT * cpt;            // step-list share-out
  auto sync = [&]() { return group_sync(&st->bar, (unsigned)cpt, a.err, lim); };
  // exclusive prefix and total over the CTAs of the group of the values
  // they left in gpw (after a barrier)
  auto group_prefix = [&]() {
    if (tid == 0) {
      int64_t p = 0, t = 0;
      for (int q = 0; q < cpt; ++q) {
        const int64_t x = *(volatile int64_t*)&gpw[q];
        if (q < r) p += x;
        t += x;
      }
      pre_sh = p;
      tot_sh = t;
    }
    __syncthreads();
  };
  for (int64_t w = wr0 + tid; w < wr1; w += GG_NT) asg[w] = 0;
  if (!sync()) return;
  int32_t* stp = a.step + base;
  int32_t* frt = a.front + base;
  int32_t* hvl = a.heavy + base;
  for (int32_t j = 0; j < k; ++j) {
    // seed: unassigned non-isolated node with the smallest hash (the row is
    // looked at only for a node that would be taken); nothing is reached yet
    const uint64_t skey = hkey(tkey, PH_GGG, (uint64_t)lvl, (uint64_t)j);
    uint64_t bh = ~0ull;
    int32_t bv = -1;
    for (int64_t v = r0 + tid; v < r1; v += GG_NT) {
      if (bit_of(asg, v)) continue;
      const uint64_t h = mix64(skey ^ (uint64_t)v);
      if ((bv < 0 || h < bh) && a.row_ptr[base + v + 1] != a.row_ptr[base + v]) {
        bh = h;
        bv = (int32_t)v;
      }
    }
    for (int64_t w = wr0 + tid; w < wr1; w += GG_NT) seen[w] = asg[w];
    for (int o = 16; o > 0; o >>= 1) {
      const uint64_t oh = __shfl_xor_sync(0xffffffffu, (unsigned long long)bh, o);
      const int32_t ov = __shfl_xor_sync(0xffffffffu, bv, o);
      if (ov >= 0 && (bv < 0 || oh < bh || (oh == bh && ov < bv))) { bh = oh; bv = ov; }
    }
    if (lane == 0) { shh[wid] = bh; shv[wid] = bv; }
    __syncthreads();
    if (tid == 0) {
      uint64_t h = ~0ull;
      int32_t v = -1;
      for (int w = 0; w < GG_NT / 32; ++w)
        if (shv[w] >= 0 && (v < 0 || shh[w] < h || (shh[w] == h && shv[w] < v))) {
          h = shh[w]; v = shv[w];
        }
      gph[r] = h;
      gpv[r] = v;
    }
    if (!sync()) return;
    if (tid == 0) {
      uint64_t h = ~0ull;
      int32_t v = -1;
      for (int q = 0; q < cpt; ++q) {
        const uint64_t qh = *(volatile uint64_t*)&gph[q];
        const int32_t qv = *(volatile int32_t*)&gpv[q];
        if (qv >= 0 && (v < 0 || qh < h || (qh == h && qv < v))) { h = qh; v = qv; }
      }
      seed_sh = v;
    }
    __syncthreads();
    const int32_t seed = seed_sh;
    if (seed < 0) break;
    if (r == 0 && tid == 0) {
      a.label[base + seed] = (int32_t)(bo + j);
      asg[seed >> 5] |= 1u << (seed & 31);
      seen[seed >> 5] |= 1u << (seed & 31);
      stp[0] = (int32_t)(base + seed);
      st->nstep = 1;
      st->nfront = 0;
      st->nnext = 0;
      st->fsum = 0;
      st->accw = 0;
      st->Wj = a.nw[base + seed];
      st->step_heavy = a.row_ptr[base + seed + 1] - a.row_ptr[base + seed] > GG_HEAVY;
      st->front_heavy = 0;
      st->next_heavy = 0;
      st->nheavy = 0;
    }
    bool ordered = false;
    if (!sync()) return;
    while (true) {
      const int32_t nstep = *(volatile int32_t*)&st->nstep;
      const bool hv_step = *(volatile int32_t*)&st->step_heavy != 0;
      int64_t fw = 0;
      // GG_ARC arcs out of the step per thread (e < 0: none; every lane of the
      // warp calls): sets their heads' seen bits; a head seen for the first
      // time is listed as reached, one list reservation per warp
      auto visit = [&](const int64_t (&e)[GG_ARC]) {
        int32_t y[GG_ARC];
        uint32_t wd[GG_ARC];
#pragma unroll
        for (int u = 0; u < GG_ARC; ++u) {
          y[u] = -1;
          if (e[u] < 0) continue;
          const int32_t h = a.col[e[u]];
          if (SCLAP_OK(h, a.N, a.err)) y[u] = (int32_t)(h - base);
        }
#pragma unroll
        for (int u = 0; u < GG_ARC; ++u) wd[u] = y[u] >= 0 ? seen[y[u] >> 5] : ~0u;
        int fresh = 0;
#pragma unroll
        for (int u = 0; u < GG_ARC; ++u) {
          const uint32_t bit = 1u << (y[u] & 31);
          if (wd[u] & bit) y[u] = -1;              // (also y < 0)
          else if (atomicOr(&seen[y[u] >> 5], bit) & bit) y[u] = -1;
          fresh += y[u] >= 0;
        }
        if (ordered) return;
        int incl = fresh;
        for (int o = 1; o < 32; o <<= 1) {
          const int z = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += z;
        }
        const int all = __shfl_sync(0xffffffffu, incl, 31);
        if (all == 0) return;
        int pos = 0;
        if (lane == 31) pos = atomicAdd(&st->nfront, all);
        pos = __shfl_sync(0xffffffffu, pos, 31) + incl - fresh;
#pragma unroll
        for (int u = 0; u < GG_ARC; ++u) {
          if (y[u] < 0) continue;
          const int64_t gy = base + y[u];
          frt[pos++] = (int32_t)gy;
          fw += a.nw[gy];
          if (a.row_ptr[gy + 1] - a.row_ptr[gy] > GG_HEAVY)
            *(volatile int32_t*)&st->front_heavy = 1;
        }
      };
      for (int64_t q0 = (int64_t)r * GG_NT; q0 < nstep; q0 += qstride) {
        const int64_t q = q0 + tid;
        int64_t rs = 0, d = 0;
        if (q < nstep) {
          const int32_t u = stp[q];
          rs = a.row_ptr[u];
          d = a.row_ptr[u + 1] - rs;
          if (hv_step && d > GG_HEAVY) {          // read by the whole group below
            hvl[atomicAdd(&st->nheavy, 1)] = u;
            d = 0;
          }
        }
        int64_t tot;
        const int64_t incl = block_incl_scan<GG_NT>(d, sh, &tot);
        st_in[tid] = (int32_t)incl;
        st_off[tid] = rs - (incl - d);
        __syncthreads();
        const int cnt = (int)min64(GG_NT, nstep - q0);
        const int32_t total = (int32_t)tot;
        const int per = min(GG_ARC, (total + GG_NT - 1) / GG_NT);
        for (int32_t c0 = 0; c0 < total; c0 += GG_NT * per) {
          // consecutive arcs per thread: one owner search for all of them
          const int32_t x0 = c0 + tid * per;
          int lo = 0, hi = cnt - 1;
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (st_in[mid] > x0) hi = mid; else lo = mid + 1;
          }
          int64_t e[GG_ARC];
#pragma unroll
          for (int u = 0; u < GG_ARC; ++u) {
            const int32_t x = x0 + u;
            e[u] = -1;
            if (u >= per || x >= total) continue;
            while (st_in[lo] <= x) ++lo;
            e[u] = st_off[lo] + x;
          }
          visit(e);
        }
        __syncthreads();
      }
      if (hv_step) {
        if (!sync()) return;                     // the heavy list is complete
        const int32_t nh = *(volatile int32_t*)&st->nheavy;
        for (int32_t hq = 0; hq < nh; ++hq) {
          const int32_t u = hvl[hq];
          const int64_t re = a.row_ptr[u + 1];
          for (int64_t e0 = a.row_ptr[u] + (int64_t)r * GG_NT; e0 < re; e0 += GG_ARC * qstride) {
            int64_t e[GG_ARC];
#pragma unroll
            for (int i = 0; i < GG_ARC; ++i) {
              const int64_t x = e0 + i * qstride + tid;
              e[i] = x < re ? x : -1;
            }
            visit(e);
          }
        }
      }
      const int64_t fwb = block_sum<GG_NT>(fw, sh);
      if (tid == 0 && fwb) atomicAdd(ull(&st->fsum), (unsigned long long)fwb);
      if (!sync()) return;
      const int64_t Wj = *(volatile int64_t*)&st->Wj;
      if (Wj >= avg) break;
      if (!ordered) {
        const int64_t fsum = *(volatile int64_t*)&st->fsum;
        const int32_t nf = *(volatile int32_t*)&st->nfront;
        if (Wj + fsum <= avg) {
          // all of them fit: they are the next step, in any order
          for (int64_t q = (int64_t)r * GG_NT + tid; q < nf; q += qstride) {
            const int64_t v = frt[q] - base;
            a.label[base + v] = (int32_t)(bo + j);
            atomicOr(&asg[v >> 5], 1u << (v & 31));
          }
          int32_t* t = stp; stp = frt; frt = t;
          if (!sync()) return;
          if (r == 0 && tid == 0) {
            st->nstep = nf;
            st->nfront = 0;
            st->fsum = 0;
            st->Wj = Wj + fsum;
            st->step_heavy = st->front_heavy;
            st->front_heavy = 0;
            st->nheavy = 0;
          }
          if (!sync()) return;
          if (nf == 0) break;
          continue;
        }
        ordered = true;
      }
      // reached unassigned nodes in id order, longest prefix that fits:
      // this CTA's range starts after the candidate weight of the ranks below
      int64_t cw = 0;
      for (int64_t v = r0 + tid; v < r1; v += GG_NT)
        if (bit_of(seen, v) && !bit_of(asg, v)) cw += a.nw[base + v];
      const int64_t cwb = block_sum<GG_NT>(cw, sh);
      if (tid == 0) gpw[r] = cwb;
      if (!sync()) return;
      group_prefix();
      const bool all_fit = Wj + tot_sh <= avg;
      int64_t carry_w = pre_sh, acc_w = 0;
      for (int64_t c0 = r0; c0 < r1; c0 += GG_NT) {
        if (!all_fit && Wj + carry_w > avg) break;          // no later candidate fits
        const int64_t v = c0 + tid;
        const bool cand = v < r1 && bit_of(seen, v) && !bit_of(asg, v);
        const int64_t wt = cand ? a.nw[base + v] : 0;
        int64_t tw;
        const int64_t iw = block_incl_scan<GG_NT>(wt, sh, &tw);
        if (cand && (all_fit || Wj + carry_w + iw <= avg)) {
          stp[atomicAdd(&st->nnext, 1)] = (int32_t)(base + v);
          acc_w += wt;
          if (a.row_ptr[base + v + 1] - a.row_ptr[base + v] > GG_HEAVY)
            *(volatile int32_t*)&st->next_heavy = 1;
        }
        carry_w += tw;
      }
      const int64_t accb = block_sum<GG_NT>(acc_w, sh);
      if (tid == 0 && accb) atomicAdd(ull(&st->accw), (unsigned long long)accb);
      if (!sync()) return;
      const int32_t ns2 = *(volatile int32_t*)&st->nnext;
      const int64_t newW = Wj + *(volatile int64_t*)&st->accw;
      for (int64_t q = (int64_t)r * GG_NT + tid; q < ns2; q += qstride) {
        const int64_t v = stp[q] - base;
        a.label[base + v] = (int32_t)(bo + j);
        atomicOr(&asg[v >> 5], 1u << (v & 31));
      }
      if (!sync()) return;
      if (r == 0 && tid == 0) {
        st->nstep = ns2;
        st->Wj = newW;
        st->nnext = 0;
        st->accw = 0;
        st->step_heavy = st->next_heavy;
        st->next_heavy = 0;
        st->front_heavy = 0;
        st->nheavy = 0;
      }
      if (!sync()) return;
      if (ns2 == 0) break;
    }
    if (r == 0 && tid == 0) a.W[bo + j] = (wgt_t)*(volatile int64_t*)&st->Wj;
    if (!sync()) return;
  }
  // water-filling of the nodes left unassigned, in id order over the trial
  int64_t rw = 0;
  for (int64_t v = r0 + tid; v < r1; v += GG_NT)
    if (!bit_of(asg, v)) rw += a.nw[base + v];
  const int64_t rwb = block_sum<GG_NT>(rw, sh);
  if (tid == 0) gpw[r] = rwb;
  if (!sync()) return;
  group_prefix();
  const int64_t R = tot_sh;
  if (R == 0) return;
  if (r == 0 && tid == 0) {
    int64_t lo = a.W[bo], hi = a.W[bo];
    for (int32_t b = 1; b < k; ++b) {
      lo = min64(lo, (int64_t)a.W[bo + b]);
      hi = max64(hi, (int64_t)a.W[bo + b]);
    }
    hi += R;
    while (lo < hi) {
      const int64_t mid = lo + (hi - lo) / 2;
      int64_t f = 0;
      for (int32_t b = 0; b < k; ++b) f += max64(0, mid - (int64_t)a.W[bo + b]);
      if (f >= R) hi = mid; else lo = mid + 1;
    }
    const int64_t L = lo;
    for (int32_t jj = 0; jj < k; ++jj) {       // insertion sort by (W, id)
      int32_t p = jj;
      while (p > 0) {
        const int32_t q = a.wforder[bo + p - 1];
        if (a.W[bo + q] > a.W[bo + jj] || (a.W[bo + q] == a.W[bo + jj] && q > jj)) {
          a.wforder[bo + p] = q;
          --p;
        } else {
          break;
        }
      }
      a.wforder[bo + p] = jj;
    }
    int64_t acc = 0;
    for (int32_t jj = 0; jj < k; ++jj) {
      a.wfA[bo + jj] = acc;
      acc += max64(0, L - (int64_t)a.W[bo + a.wforder[bo + jj]]);
    }
  }
  if (!sync()) return;
  int64_t carry = pre_sh;
  for (int64_t v0 = r0; v0 < r1; v0 += GG_NT) {
    const int64_t v = v0 + tid;
    const bool left = v < r1 && !bit_of(asg, v);
    const int64_t wt = left ? a.nw[base + v] : 0;
    int64_t tw;
    const int64_t iw = block_incl_scan<GG_NT>(wt, sh, &tw);
    if (left) {
      const int64_t p = carry + iw - wt;
      int32_t lo = 0, hi = k - 1;               // last j with A[j] <= p
      while (lo < hi) {
        const int32_t mid = (lo + hi + 1) >> 1;
        if (a.wfA[bo + mid] <= p) lo = mid; else hi = mid - 1;
      }
      const int32_t b = a.wforder[bo + lo];
      a.label[base + v] = (int32_t)(bo + b);
      atomicAdd(&a.W[bo + b], (wgt_t)wt);
    }
    carry += tw;
  }
}

// Twice the cut of every slot (every edge is met from both ends).  The arcs
// are streamed in storage order (arcs.cuh), so a hub's row and an empty
// graph cost what their arcs cost; per tile a thread's eight label gathers
// are in flight together, a slot's sum stays in a register until the CTA
// leaves the slot, then one atomic adds it.
// Bounded by the label gathers through L1 and L2 (55-68 % busy).  Measured
// on R-MAT 2^21 nodes, 56 M weighted arcs: 743 -> 310 us (a warp per 32 rows
// plus a queue of long rows before); the 512-graph batch's trial and final
// cuts 1.74 -> 1.12 ms.  Five CTAs per SM: for six it spills 72 bytes a thread
// (R-MAT 2^24 nodes 3.76 ms, five 3.16, four 3.38).
constexpr int CUT_CTAS = 5;
template <int R>
__global__ void __launch_bounds__(AT_NT, CUT_CTAS) k_slot_cut(const int64_t* __restrict__ row_ptr,
                                                    const int32_t* __restrict__ col,
                                                    const int32_t* __restrict__ ew,
                                                    const int64_t* __restrict__ noff,
                                                    const int64_t* __restrict__ aoff,
                                                    int32_t nslots, int64_t N, int64_t M,
                                                    const int32_t* __restrict__ label,
                                                    int64_t* __restrict__ cut2) {
  __shared__ int32_t sh_end[R * AT_V];
  __shared__ unsigned long long sh_sum[AT_NT / 32];
  int64_t lo, hi;
  arc_share(M, &lo, &hi);
  while (lo < hi) {
    const int32_t s = nslots > 1 ? slot_of(aoff, nslots, lo) : 0;
    const int64_t end = nslots > 1 ? min64(hi, aoff[s + 1]) : hi;
    unsigned long long acc = 0;
    for_arc_tiles<R>(row_ptr, nslots > 1 ? noff[s] : 0, nslots > 1 ? noff[s + 1] : N, lo, end, col,
                     ew, M, sh_end, [&](const ArcTile& t, int64_t, int32_t) {
      int32_t a[AT_PER], b[AT_PER];
#pragma unroll
      for (int i = 0; i < AT_PER; ++i) {
        a[i] = t.v[i] >= 0 ? label[t.v[i]] : 0;
        b[i] = t.v[i] >= 0 ? label[t.c[i]] : 0;
      }
#pragma unroll
      for (int i = 0; i < AT_PER; ++i) acc += a[i] != b[i] ? (unsigned long long)t.w[i] : 0ull;
    });
    const unsigned long long tot = cta_sum(acc, sh_sum);
    if (threadIdx.x == 0 && tot) atomicAdd(ull(&cut2[s]), tot);
    lo = end;
  }
}

// Twice the cuts of the trials of every graph at once.  A graph's trials share
// its structure, so its arcs are streamed once, not once per trial, and the
// block ids of a node in TC of the trials lie side by side in one 16-byte word
// (blocks fit a byte): an arc gathers one word for all of them instead of one
// label per trial.  Bound by streaming the arcs (8 bytes each, once per TC
// trials).  16 trials, per-trial streams -> one: a web graph of 2^24 nodes
// 28.0 -> 3.2 ms, an R-MAT graph of 2^22 nodes 2.54 -> 0.34 ms, 512 small
// graphs 0.73 -> 0.19 ms.
constexpr int TC = 16;
constexpr int64_t TC_MIN_ARCS = (int64_t)4 << 20;   // over all trials
struct TrialCut {
  const int64_t* noff;     // slots (B * T): first node, first arc, first block
  const int64_t* aoff;
  const int64_t* boff;
  const int64_t* nbase;    // [B + 1] first packed word of each graph
  const int64_t* abase;    // [B + 1] arcs of the graphs, back to back
  int32_t B, T, t0, tn;    // graphs, trials, and the trials of this pass
};
__global__ void __launch_bounds__(256) k_pack_trials(TrialCut a, const int32_t* __restrict__ label,
                                                     uint4* __restrict__ pk) {
  const int64_t n = a.nbase[a.B];
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n;
       x += (int64_t)gridDim.x * blockDim.x) {
    const int32_t g = slot_of(a.nbase, a.B, x);
    // a graph's slots are equally long in nodes and blocks
    const int64_t s0 = (int64_t)g * a.T, n0 = a.noff[s0], b0 = a.boff[s0];
    const int64_t nd = a.noff[s0 + 1] - n0;
    const int32_t k = (int32_t)(a.boff[s0 + 1] - b0);
    const int32_t* l = label + n0 + a.t0 * nd + (x - a.nbase[g]);
    uint32_t b[TC], w[4] = {0, 0, 0, 0};
#pragma unroll
    for (int t = 0; t < TC; ++t) b[t] = t < a.tn ? (uint32_t)l[t * nd] : 0u;
#pragma unroll
    for (int t = 0; t < TC; ++t)
      if (t < a.tn)
        w[t >> 2] |= (b[t] - (uint32_t)(b0 + (int64_t)(a.t0 + t) * k)) << (8 * (t & 3));
    pk[x] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}
__global__ void __launch_bounds__(AT_NT, 2) k_trial_cut(TrialCut a, const int64_t* __restrict__ row_ptr,
                                                        const int32_t* __restrict__ col,
                                                        const int32_t* __restrict__ ew, int64_t M,
                                                        const uint4* __restrict__ pk,
                                                        int64_t* __restrict__ cut2) {
  __shared__ int32_t sh_end[AT_V];
  __shared__ unsigned long long sh_sum[TC];
  const int tid = threadIdx.x;
  int64_t lo, hi;
  arc_share(a.abase[a.B], &lo, &hi);
  while (lo < hi) {
    const int32_t g = slot_of(a.abase, a.B, lo);
    const int64_t end = min64(hi, a.abase[g + 1]);
    const int64_t s0 = (int64_t)g * a.T, first = a.aoff[s0] - a.abase[g];
    const int64_t n0 = a.noff[s0];
    const uint4* words = pk + a.nbase[g];
    unsigned long long acc[TC];
#pragma unroll
    for (int t = 0; t < TC; ++t) acc[t] = 0;
    if (tid < TC) sh_sum[tid] = 0;
    for_arc_tiles(row_ptr, n0, a.noff[s0 + 1], lo + first, end + first, col, ew, M, sh_end,
                  [&](const ArcTile& t, int64_t, int32_t) {
#pragma unroll
      for (int h = 0; h < AT_PER; h += 4) {
        uint4 x[4], y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const bool in = t.v[h + i] >= 0;
          x[i] = in ? words[t.v[h + i] - n0] : make_uint4(0, 0, 0, 0);
          y[i] = in ? words[t.c[h + i] - n0] : make_uint4(0, 0, 0, 0);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t d[4] = {x[i].x ^ y[i].x, x[i].y ^ y[i].y, x[i].z ^ y[i].z, x[i].w ^ y[i].w};
          const unsigned long long w = (unsigned long long)t.w[h + i];
#pragma unroll
          for (int q = 0; q < TC; ++q) acc[q] += (d[q >> 2] >> (8 * (q & 3))) & 0xffu ? w : 0ull;
        }
      }
    });
    __syncthreads();
#pragma unroll
    for (int t = 0; t < TC; ++t) {
      unsigned long long v = acc[t];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if ((tid & 31) == 0 && v) atomicAdd(&sh_sum[t], v);
    }
    __syncthreads();
    if (tid < a.tn && sh_sum[tid]) atomicAdd(ull(&cut2[s0 + a.t0 + tid]), sh_sum[tid]);
    __syncthreads();
    lo = end;
  }
}

// Best trial of each task (a graph's trials of one group): least overload,
// then least cut; it replaces the graph's best so far only if better (the
// groups run in trial order, so the first best trial wins ties).  take[i] =
// the task's trial to copy out, or -1.
__global__ void k_select_best(const SelectTask* __restrict__ tasks, int32_t ntasks,
                              const int64_t* __restrict__ cut2, const wgt_t* __restrict__ ip_W,
                              const int64_t* __restrict__ ip_boff, int32_t* __restrict__ best,
                              int64_t* __restrict__ ipcut, int64_t* __restrict__ rb_ov,
                              int32_t* __restrict__ take) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntasks) return;
  const SelectTask t = tasks[i];
  int64_t bo = -1, bc = -1;
  int32_t bt = -1;
  for (int32_t tr = 0; tr < t.trials; ++tr) {
    const int64_t slot = t.slot0 + tr;
    int64_t mx = 0;
    for (int32_t b = 0; b < t.k; ++b) mx = max64(mx, (int64_t)ip_W[ip_boff[slot] + b]);
    const int64_t ov = max64(0, mx - t.Lmax);
    const int64_t c = cut2[slot] / 2;
    if (bt < 0 || ov < bo || (ov == bo && c < bc)) { bo = ov; bc = c; bt = tr; }
  }
  const bool tk = best[t.g] < 0 || bo < rb_ov[t.g] || (bo == rb_ov[t.g] && bc < ipcut[t.g]);
  if (tk) {
    best[t.g] = t.trial0 + bt;
    ipcut[t.g] = bc;
    rb_ov[t.g] = bo;
  }
  take[i] = tk ? bt : -1;
}

// Copies the taken trial's blocks out: tasks along y, chunks of SC_CH nodes
// along x.
constexpr int64_t SC_CH = 65536;
__global__ void k_copy_best(const SelectTask* __restrict__ tasks, const int32_t* __restrict__ take,
                            const int64_t* __restrict__ ip_noff, const int64_t* __restrict__ ip_boff,
                            const int32_t* __restrict__ ip_label, const wgt_t* __restrict__ ip_W,
                            wgt_t* __restrict__ Wg) {
  const int32_t bt = take[blockIdx.y];
  if (bt < 0) return;
  const SelectTask t = tasks[blockIdx.y];
  const int64_t slot = t.slot0 + bt;
  const int64_t src = ip_noff[slot], sbo = ip_boff[slot];
  const int64_t v1 = min64(((int64_t)blockIdx.x + 1) * SC_CH, t.n);
  for (int64_t v = (int64_t)blockIdx.x * SC_CH + threadIdx.x; v < v1; v += blockDim.x) {
    int64_t d = v;
    if (t.rank) {
      const int64_t r0 = t.rank[t.dst_n0 + v];
      if (t.rank[t.dst_n0 + v + 1] == r0) { t.dst_blk[t.dst_n0 + v] = -1; continue; }
      d = r0 - t.rbase;
    }
    t.dst_blk[t.dst_n0 + v] = (int32_t)(t.g_boff + (ip_label[src + d] - sbo));
  }
  if (blockIdx.x == 0)
    for (int32_t b = threadIdx.x; b < t.k; b += blockDim.x) Wg[t.g_boff + b] = ip_W[sbo + b];
}

__global__ void k_project(const int32_t* __restrict__ cmap, const int32_t* __restrict__ cblk,
                          int32_t* __restrict__ fblk, int64_t N) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t c = cmap[v];
    if (c >= 0) fblk[v] = cblk[c];
  }
}

__global__ void k_lift_blocks(const int32_t* __restrict__ cmap, const int32_t* __restrict__ fblk,
                              int32_t* __restrict__ cblk, int64_t N) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t c = cmap[v];
    if (c >= 0) cblk[c] = fblk[v];
  }
}

// Block weights from scratch.  With at most BW_SH blocks a CTA sums its
// nodes in shared memory first and adds each block once: the blocks are few,
// so one global atomic per node serialised on a handful of addresses.
// 2^20 nodes, 16 blocks: 175 -> 14 us.
constexpr int BW_SH = 2048;
__global__ void __launch_bounds__(256) k_block_weights(const int32_t* __restrict__ label,
                                                       const int32_t* __restrict__ nw, int64_t N,
                                                       wgt_t* __restrict__ W, int64_t nlabels) {
  __shared__ int32_t sh[BW_SH];
  const bool few = nlabels <= BW_SH;
  if (few) {
    for (int b = threadIdx.x; b < nlabels; b += blockDim.x) sh[b] = 0;
    __syncthreads();
  }
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N;
       v += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(few ? &sh[label[v]] : &W[label[v]], (wgt_t)wat(nw, v));
  if (few) {
    __syncthreads();
    for (int b = threadIdx.x; b < nlabels; b += blockDim.x)
      if (sh[b]) atomicAdd(&W[b], sh[b]);
  }
}

__global__ void k_isolated(const int64_t* __restrict__ row_ptr, const int32_t* __restrict__ nw,
                           int64_t N, uint8_t* __restrict__ flags, int32_t* __restrict__ iso_w) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < N;
       v += (int64_t)gridDim.x * blockDim.x) {
    const bool has = row_ptr[v + 1] > row_ptr[v];
    flags[v] = has ? 1 : 0;
    iso_w[v] = has ? 0 : wat(nw, v);
  }
}

// One thread per graph: fill level L (smallest L with sum_b max(0, L - W_b)
// >= R), blocks ordered by (weight, id), and the start of each block's
// stretch of free capacity below L.
__global__ void k_wf_setup(const FillTask* __restrict__ tasks, int ntasks, const wgt_t* Wg,
                           int32_t* order, int64_t* A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntasks) return;
  const FillTask t = tasks[i];
  const int64_t R = t.iso_prefix[t.n0 + t.n] - t.iso_prefix[t.n0];
  if (R == 0) return;
  const wgt_t* W = Wg + t.g_boff;
  int64_t lo = W[0], hi = W[0];
  for (int32_t b = 1; b < t.k; ++b) { lo = min64(lo, (int64_t)W[b]); hi = max64(hi, (int64_t)W[b]); }
  hi += R;
  while (lo < hi) {
    const int64_t mid = lo + (hi - lo) / 2;
    int64_t f = 0;
    for (int32_t b = 0; b < t.k; ++b) f += max64(0, mid - (int64_t)W[b]);
    if (f >= R) hi = mid; else lo = mid + 1;
  }
  int32_t* ord = order + t.g_boff;
  for (int32_t j = 0; j < t.k; ++j) {
    int32_t p = j;
    while (p > 0) {
      const int32_t q = ord[p - 1];
      if (W[q] > W[j] || (W[q] == W[j] && q > j)) { ord[p] = q; --p; } else break;
    }
    ord[p] = j;
  }
  int64_t acc = 0;
  for (int32_t j = 0; j < t.k; ++j) {
    A[t.g_boff + j] = acc;
    acc += max64(0, lo - (int64_t)W[ord[j]]);
  }
}

// The block weights are summed per CTA first (up to WF_SH blocks): one global
// atomic per isolated node serialised on the few lightest blocks
// (R-MAT 2^24 nodes, k = 16: 4.41 ms -> 60 us).
constexpr int WF_SH = 1024;
__global__ void __launch_bounds__(256) k_wf_assign(const FillTask* __restrict__ tasks, wgt_t* Wg,
                                                   const int32_t* __restrict__ order,
                                                   const int64_t* __restrict__ A) {
  __shared__ int32_t sh[WF_SH];
  const FillTask t = tasks[blockIdx.y];
  const int64_t base = t.iso_prefix[t.n0];
  if (t.iso_prefix[t.n0 + t.n] == base) return;    // no isolated node
  const bool few = t.k <= WF_SH;
  if (few) {
    for (int b = threadIdx.x; b < t.k; b += blockDim.x) sh[b] = 0;
    __syncthreads();
  }
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < t.n;
       v += (int64_t)gridDim.x * blockDim.x) {
    if (t.blk[t.n0 + v] >= 0) continue;
    const int64_t p = t.iso_prefix[t.n0 + v] - base;
    int32_t lo = 0, hi = t.k - 1;   // last j with A[j] <= p
    while (lo < hi) {
      const int32_t mid = (lo + hi + 1) >> 1;
      if (A[t.g_boff + mid] <= p) lo = mid; else hi = mid - 1;
    }
    const int32_t b = order[t.g_boff + lo];
    t.blk[t.n0 + v] = (int32_t)(t.g_boff + b);
    atomicAdd(few ? &sh[b] : &Wg[t.g_boff + b], (wgt_t)wat(t.nw, t.n0 + v));
  }
  if (few) {
    __syncthreads();
    for (int b = threadIdx.x; b < t.k; b += blockDim.x)
      if (sh[b]) atomicAdd(&Wg[t.g_boff + b], sh[b]);
  }
}

}  // namespace

void isolated_flags(const int64_t* row_ptr, const int32_t* nw, int64_t N, uint8_t* flags,
                    int32_t* iso_w, cudaStream_t s) {
  if (N <= 0) return;
  k_isolated<<<grid_for(N, 256, (int64_t)num_sms() * 16), 256, 0, s>>>(row_ptr, nw, N, flags, iso_w); SCLAP_NOTE_LAUNCH("k_isolated");
  SCLAP_LAUNCH_CHECK();
}

void waterfill_isolated(const std::vector<FillTask>& tasks, wgt_t* Wg, int64_t Ktot,
                        cudaStream_t s) {
  if (tasks.empty()) return;
  DevBuf<FillTask> d(tasks.size(), s);
  d.upload(tasks);
  DevBuf<int32_t> order(std::max<int64_t>(Ktot, 1), s);
  DevBuf<int64_t> A(std::max<int64_t>(Ktot, 1), s);
  const int nt = (int)tasks.size();
  k_wf_setup<<<(nt + 127) / 128, 128, 0, s>>>(d.p, nt, Wg, order.p, A.p); SCLAP_NOTE_LAUNCH("k_wf_setup");
  int64_t mx = 1;
  for (const auto& t : tasks) mx = std::max(mx, t.n);
  const int64_t per_task = std::max<int64_t>(64, (int64_t)num_sms() * 8 / nt);
  for (int t0 = 0; t0 < nt; t0 += 65535) {
    dim3 grid(grid_for(mx, 256, per_task), (unsigned)std::min(65535, nt - t0));
    k_wf_assign<<<grid, 256, 0, s>>>(d.p + t0, Wg, order.p, A.p); SCLAP_NOTE_LAUNCH("k_wf_assign");
  }
  SCLAP_LAUNCH_CHECK();
}

void ip_replicate(const std::vector<CopyTask>& tasks, int64_t* row_ptr, int32_t* col,
                  int32_t* ew, int32_t* nw, int64_t M_total, cudaStream_t s,
                  int64_t N_total_override) {
  if (tasks.empty()) return;
  DevBuf<CopyTask> d(tasks.size(), s);
  d.upload(tasks);
  int64_t mx = 1, copies = 1;
  for (const auto& t : tasks) {
    mx = std::max(mx, std::max(t.n, t.m));
    copies = std::max<int64_t>(copies, t.copies);
  }
  // at least 64 CTAs per task, more when few tasks would leave SMs idle; short
  // segments share out the copies until the chip has eight CTAs per SM
  const int64_t want = (int64_t)num_sms() * 8, nt = (int64_t)tasks.size();
  const int gx = grid_for(mx, RP_NT * RP_PER, std::max<int64_t>(64, want / nt));
  const unsigned nz = (unsigned)std::min<int64_t>(copies, std::max<int64_t>(1, want / (gx * nt)));
  for (size_t t0 = 0; t0 < tasks.size(); t0 += 65535) {
    const unsigned ny = (unsigned)std::min<size_t>(65535, tasks.size() - t0);
    k_replicate<<<dim3(gx, ny, nz), RP_NT, 0, s>>>(d.p + t0, row_ptr, col, ew, nw); SCLAP_NOTE_LAUNCH("k_replicate");
  }
  int64_t Ntot = 0;
  for (const auto& t : tasks) {
    const int64_t nd = t.rank ? 0 : t.n;   // renumbered tasks: caller passes dst end below
    Ntot = std::max(Ntot, t.dst_n0 + nd);
  }
  if (N_total_override >= 0) Ntot = N_total_override;
  k_set_i64<<<1, 1, 0, s>>>(row_ptr + Ntot, M_total); SCLAP_NOTE_LAUNCH("k_set_i64");
  SCLAP_LAUNCH_CHECK();
}

void ggg_trials(const GGGArgs& a_in, const std::vector<int64_t>& noff,
                const std::vector<int32_t>& nlab, cudaStream_t s) {
  if (a_in.nslots <= 0) return;
  const int32_t S = a_in.nslots;
  // longest processing time first: trial slots by node count, descending
  std::vector<int32_t> order(S);
  for (int32_t i = 0; i < S; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
    return noff[x + 1] - noff[x] > noff[y + 1] - noff[y];
  });
  // bitmaps (cleared by the kernels): the words of every trial
  const int64_t bwords = ggg_word0(noff[S], S) + 1;
  DevBuf<uint32_t> bits((size_t)(2 * bwords), s);
  DevBuf<int32_t> d_order(S, s), d_next(1, s);
  d_order.upload(order);
  d_next.zero();
  GGGArgs a = a_in;
  a.order = d_order.p;
  a.next = d_next.p;
  a.asg = bits.p;
  a.seen = bits.p + bwords;
  // a trial is a chain of small steps, so the kernel is bound by how many
  // trials are in flight: small CTAs when the trials outnumber the resident
  // 512-thread CTAs
  int few_per_sm = 0, many_per_sm = 0;
  SCLAP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&few_per_sm, k_ggg<GNT_FEW>, GNT_FEW, 0));
  SCLAP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&many_per_sm, k_ggg<GNT_MANY>, GNT_MANY, 0));
  const int64_t few_resident = (int64_t)num_sms() * std::max(few_per_sm, 1);
  const int64_t many_resident = (int64_t)num_sms() * std::max(many_per_sm, 1);
  // few trials of large blocks: a group of CTAs per trial (the resident
  // CTAs shared out, at most 256 per trial, and only when every trial gets
  // at least 4).  A growth step
  // costs the group a few barriers, so the groups pay off only when the
  // blocks are large: measured faster on R-MAT scale 22 at k = 2 and 8 and
  // on scale 25 at k = 16 (1149 -> 369 ms), slower on scale 22 at k = 32
  // and 64, and the same gate cannot separate them at 2^16 or 2^17 nodes per
  // block (scale 22, k = 8 fell below 2^15 as well); the gate is 2^14
  // nodes per block on average in some trial.
  int group_per_sm = 0;
  SCLAP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&group_per_sm, k_ggg_group, GG_NT, 0));
  const int64_t group_resident = (int64_t)num_sms() * std::max(group_per_sm, 1);
  const int64_t cpt = std::min<int64_t>(256, group_resident / S);
  int64_t per_block = 0;
  for (int32_t i = 0; i < S; ++i)
    per_block = std::max(per_block, (noff[i + 1] - noff[i]) / std::max<int32_t>(1, nlab[i]));
  if (cpt >= 4 && per_block >= ((int64_t)1 << 14)) {
    DevBuf<GroupState> gs(S, s);
    DevBuf<uint64_t> ph(S * cpt, s);
    DevBuf<int32_t> pv(S * cpt, s);
    DevBuf<int64_t> pw(S * cpt, s);
    gs.zero();
    k_first_blocks<<<dim3(grid_for(noff[S] / S, 256 * 4, 256), (unsigned)S), 256, 0, s>>>(a); SCLAP_NOTE_LAUNCH("k_first_blocks");
    launch_coop(k_ggg_group, (unsigned)(S * cpt), GG_NT, 0, s, a, (int32_t)cpt, gs.p, ph.p, pv.p,
                pw.p, wait_limit()); SCLAP_NOTE_LAUNCH("k_ggg_group");
    SCLAP_LAUNCH_CHECK();
    return;
  }
  if (S > few_resident) {
    k_ggg<GNT_MANY><<<(unsigned)std::min<int64_t>(S, many_resident), GNT_MANY, 0, s>>>(a); SCLAP_NOTE_LAUNCH("k_ggg");
  } else {
    k_ggg<GNT_FEW><<<(unsigned)std::min<int64_t>(S, few_resident), GNT_FEW, 0, s>>>(a); SCLAP_NOTE_LAUNCH("k_ggg");
  }
  SCLAP_LAUNCH_CHECK();
}

void slot_cut(const LevelView& lv, const int32_t* label, int64_t* cut2, cudaStream_t s) {
  if (lv.M <= 0) return;
  (rows_short(lv.M, lv.N) ? k_slot_cut<SHORT_ROWS> : k_slot_cut<1>)<<<arc_grid(lv.M, lv.N, CUT_CTAS), AT_NT, 0, s>>>(lv.row_ptr, lv.col, lv.ew, lv.noff, lv.aoff,
                                                 lv.nslots, lv.N, lv.M, label, cut2); SCLAP_NOTE_LAUNCH("k_slot_cut");
  SCLAP_LAUNCH_CHECK();
}

void trial_cuts(const LevelView& lv, int B, int T, const std::vector<int64_t>& noff,
                const std::vector<int64_t>& aoff, const int64_t* d_boff, int32_t max_k,
                const int32_t* label, int64_t* cut2, cudaStream_t s) {
  // One trial gains nothing, more than 256 blocks do not fit a byte.  Short
  // batches are launch-bound: per-trial streams take about 10 us per million
  // arcs, packing costs one more launch and an upload (1.2 M arcs: 18 us
  // against 36; 80 M: 730 against 190).
  if (T < 2 || max_k > 256 || lv.M < TC_MIN_ARCS) {
    slot_cut(lv, label, cut2, s);
    return;
  }
  std::vector<int64_t> base(2 * (B + 1), 0);
  for (int g = 0; g < B; ++g) {
    const size_t q = (size_t)g * T;
    base[g + 1] = base[g] + noff[q + 1] - noff[q];
    base[B + 1 + g + 1] = base[B + 1 + g] + aoff[q + 1] - aoff[q];
  }
  const int64_t n = base[B], m = base[2 * B + 1];
  if (m <= 0) return;
  DevBuf<int64_t> d_base(base.size(), s);
  d_base.upload(base);
  DevBuf<uint4> pk((size_t)n, s);
  TrialCut a{lv.noff, lv.aoff, d_boff, d_base.p, d_base.p + B + 1, B, T, 0, 0};
  for (a.t0 = 0; a.t0 < T; a.t0 += TC) {
    a.tn = std::min(TC, T - a.t0);
    k_pack_trials<<<grid_for(n, 256, (int64_t)num_sms() * 16), 256, 0, s>>>(a, label, pk.p); SCLAP_NOTE_LAUNCH("k_pack_trials");
    k_trial_cut<<<arc_grid(m, n, 2), AT_NT, 0, s>>>(a, lv.row_ptr, lv.col, lv.ew, lv.M, pk.p, cut2); SCLAP_NOTE_LAUNCH("k_trial_cut");
  }
  SCLAP_LAUNCH_CHECK();
}

void ip_select_copy(const std::vector<SelectTask>& tasks, const int64_t* cut2,
                    const wgt_t* ip_W, const int64_t* ip_noff, const int64_t* ip_boff,
                    const int32_t* ip_label, wgt_t* Wg, int32_t* best, int64_t* ipcut,
                    int64_t* rb_ov, cudaStream_t s) {
  if (tasks.empty()) return;
  const int32_t nt = (int32_t)tasks.size();
  DevBuf<SelectTask> d(nt, s);
  DevBuf<int32_t> take(nt, s);
  d.upload(tasks);
  k_select_best<<<(nt + 127) / 128, 128, 0, s>>>(d.p, nt, cut2, ip_W, ip_boff, best, ipcut, rb_ov,
                                                 take.p); SCLAP_NOTE_LAUNCH("k_select_best");
  int64_t mx = 1;
  for (const auto& t : tasks) mx = std::max(mx, t.n);
  for (int32_t t0 = 0; t0 < nt; t0 += 65535) {
    dim3 grid((unsigned)((mx + SC_CH - 1) / SC_CH), (unsigned)std::min(65535, nt - t0));
    k_copy_best<<<grid, 256, 0, s>>>(d.p + t0, take.p + t0, ip_noff, ip_boff, ip_label, ip_W, Wg); SCLAP_NOTE_LAUNCH("k_copy_best");
  }
  SCLAP_LAUNCH_CHECK();
}

void project(const int32_t* cmap, const int32_t* coarse_blk, int32_t* fine_blk, int64_t N,
             cudaStream_t s) {
  if (N <= 0) return;
  k_project<<<grid_for(N, 256, (int64_t)num_sms() * 16), 256, 0, s>>>(cmap, coarse_blk,
                                                                      fine_blk, N); SCLAP_NOTE_LAUNCH("k_project");
  SCLAP_LAUNCH_CHECK();
}

void lift_blocks(const int32_t* cmap, const int32_t* fine_blk, int32_t* coarse_blk, int64_t N,
                 cudaStream_t s) {
  if (N <= 0) return;
  k_lift_blocks<<<grid_for(N, 256, (int64_t)num_sms() * 16), 256, 0, s>>>(cmap, fine_blk,
                                                                          coarse_blk, N); SCLAP_NOTE_LAUNCH("k_lift_blocks");
  SCLAP_LAUNCH_CHECK();
}

void block_weights(const int32_t* label, const int32_t* nw, int64_t N, wgt_t* W, int64_t nlabels,
                   cudaStream_t s) {
  if (N <= 0) return;
  k_block_weights<<<grid_for(N, 256 * 8, (int64_t)num_sms() * 8), 256, 0, s>>>(label, nw, N, W,
                                                                             nlabels); SCLAP_NOTE_LAUNCH("k_block_weights");
  SCLAP_LAUNCH_CHECK();
}

}  // namespace sclap
