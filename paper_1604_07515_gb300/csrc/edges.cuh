// The edges of a frontier dealt to warps: every warp takes 32 * IT consecutive
// edges of the concatenated adjacency lists at a time.
#pragma once

#include "common.cuh"

namespace lgc {

// The first index of a[0, n) (non-decreasing) whose entry exceeds x, found
// by all 32 lanes of a warp (the same result in each): every step probes the
// last entry of 32 equal chunks of the range and keeps the chunk where the
// entries start to exceed x, so a search over n entries takes about
// log32(n) dependent loads instead of log2(n).
__device__ inline int64_t warp_upper_bound(const int64_t* a, int64_t n, int64_t x) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n;  // the answer lies in [lo, hi]
  while (hi - lo > 32) {
    const int64_t step = (hi - lo + 31) / 32;
    const int64_t pos = lo + (int64_t)(lane + 1) * step - 1;
    const bool le = pos < hi && a[pos] <= x;  // true on a prefix of the lanes
    const int c = __popc(__ballot_sync(0xffffffffu, le));
    lo += (int64_t)c * step;
    if (lo >= hi) return hi;
    hi = min(hi, lo + step);
  }
  const bool le = lo + lane < hi && a[lo + lane] <= x;
  return lo + __popc(__ballot_sync(0xffffffffu, le));
}

// Calls fn(src, at) with each lane's edges e0 + 32 k + lane of a tile of
// 32 * IT edges: their sources src[k] (-1 past the end) and their places at[k]
// in the adjacency.  epos: the sources' first edges (exclusive prefix sums of
// their degrees, all at least 1), foff: their lists' starts.  A tile's first
// source comes from a search; from there on the sources that start within the
// next 32 edges are one load and one OR-reduction away.  No shared memory and
// no block barriers: staging tiles of 1024 edges through shared memory, with a
// binary search per edge, had the bulk push wait on barriers and shared memory
// half of the time.
template <int IT, class Fn>
__device__ inline void warp_edges(const int64_t* epos, const int64_t* foff, int64_t nf, int64_t E,
                                  int64_t warp, int64_t nwarps, Fn&& fn) {
  const int lane = threadIdx.x & 31;
  for (int64_t e0 = warp * 32 * IT; e0 < E; e0 += nwarps * 32 * IT) {
    int64_t j = max((int64_t)0, warp_upper_bound(epos, nf, e0) - 1);
    int64_t bj = foff[j] - epos[j];
    int32_t src[IT];
    int64_t at[IT];
#pragma unroll
    for (int k = 0; k < IT; k++) {
      const int64_t eb = e0 + 32 * k;
      const bool in = j + 1 + lane < nf;
      const int64_t st = in ? epos[j + 1 + lane] : INT64_MAX;
      const int64_t bw = in ? foff[j + 1 + lane] - st : 0;
      const uint32_t rel = (uint32_t)min(st - eb, (int64_t)32);
      const unsigned m = __reduce_or_sync(0xffffffffu, rel < 32u ? 1u << rel : 0u);
      const int i = __popc(m & (0xffffffffu >> (31 - lane)));  // sources past j
      const int64_t bs = __shfl_sync(0xffffffffu, bw, max(i - 1, 0));
      src[k] = eb + lane < E ? (int32_t)(j + i) : -1;
      at[k] = (i ? bs : bj) + eb + lane;
      const int all = __popc(m);
      const int64_t bl = __shfl_sync(0xffffffffu, bw, max(all - 1, 0));
      bj = all ? bl : bj;
      j += all;
    }
    fn(src, at);
  }
}

// ---------------------------------------------------------------------------
// Hot destinations.  Adds to one address are served one after another, about
// 2.9 ns an FP64 add: a round that pushes 7M edges of an R-MAT graph adds
// 45,583 of them to its hub, which took 131 us, whatever the other edges
// needed (about 55).  The adds to the graph's kHot vertices of highest degree
// are summed per thread, then per block, and reach memory once per block.
// ---------------------------------------------------------------------------
struct HotSum {
  double a[kHot] = {};
  unsigned any = 0;
};

// The edges with w in H join S and become w = -1 (all lanes call it).
template <int IT>
__device__ inline void hot_take(const HotSet& H, HotSum& S, int32_t (&w)[IT],
                                const double (&sh)[IT]) {
#pragma unroll
  for (int k = 0; k < IT; k++) {
    bool hit = false;
#pragma unroll
    for (int h = 0; h < kHot; h++) hit = hit || w[k] == H.v[h];
    if (!__any_sync(0xffffffffu, hit)) continue;
#pragma unroll
    for (int h = 0; h < kHot; h++)
      if (w[k] == H.v[h]) {
        S.a[h] = S.a[h] + sh[k];
        S.any |= 1u << h;
      }
    if (hit) w[k] = -1;
  }
}

// Every thread of the block calls it; thread h < kHot calls add(h, sum) if any
// thread met H.v[h].
template <int WARPS, class Add>
__device__ inline void hot_flush(const HotSum& S, Add&& add) {
  __shared__ double s_hot[WARPS][kHot];
  __shared__ unsigned s_any;
  const unsigned any = __syncthreads_or(S.any != 0);
  if (!any) return;
  if (threadIdx.x == 0) s_any = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const unsigned met = __reduce_or_sync(0xffffffffu, S.any);
#pragma unroll
  for (int h = 0; h < kHot; h++) {
    double x = S.a[h];
    if ((met >> h) & 1u)  // the sums of warps that met it (FP64 adds are dear)
      for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) s_hot[threadIdx.x >> 5][h] = x;
  }
  if (lane == 0 && met) atomicOr(&s_any, met);
  __syncthreads();
  if (threadIdx.x < kHot && ((s_any >> threadIdx.x) & 1u)) {
    double x = 0.0;
    for (int k = 0; k < WARPS; k++)
      if (s_hot[k][threadIdx.x] != 0.0) x += s_hot[k][threadIdx.x];
    add((int)threadIdx.x, x);
  }
}

}  // namespace lgc
