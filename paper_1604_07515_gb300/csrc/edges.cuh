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

// The sources of a warp's consecutive edges: a window of the 32 sources after
// source j, their first edges one per lane.  While the window's last source
// starts past an edge, the edge's source is known from the window: a tile of
// 256 edges of an R-MAT frontier (70 a source) takes one load.
// start(i), i < nf: the first edge of source i; base(i): its list's start less
// that.  Every source has edges: the OR of find counts those with one first
// edge once.  Sources without any (lgc_graph::sinks) are put behind the others,
// all starting at the end, by the caller.
template <class Start, class Base>
struct EdgeWindow {
  int64_t j, bj;  // the source the window follows, its base
  int64_t st, bw; // this lane's: source j + 1 + lane
  int64_t nf;
  Start start;
  Base base;
  __device__ EdgeWindow(int64_t first, int64_t n, Start s, Base b) : nf(n), start(s), base(b) {
    load(first);
  }
  __device__ void load(int64_t first) {
    const int64_t i = first + 1 + (threadIdx.x & 31);
    j = first;
    bj = base(first);
    st = i < nf ? start(i) : INT64_MAX;
    bw = i < nf ? base(i) : 0;
  }
  // Lane l's edge eb + l (eb: the same in every lane, not below the last
  // call's): its source, and its list's base.
  __device__ int64_t find(int64_t eb, int64_t* b) {
    const int lane = threadIdx.x & 31;
    for (;;) {
      const int below = __popc(__ballot_sync(0xffffffffu, st < eb));
      const int64_t rel = st - eb;
      const unsigned m =
          __reduce_or_sync(0xffffffffu, rel >= 0 && rel < 32 ? 1u << (int)rel : 0u);
      const int all = below + __popc(m);  // sources of the window that start by eb + 31
      if (all == 32 && below > 0) {  // sources past the window may, too
        load(j + below);  // the last one that starts before eb: at most 32 start by eb + 31
        continue;
      }
      const int i = below + __popc(m & (0xffffffffu >> (31 - lane)));
      const int64_t bs = __shfl_sync(0xffffffffu, bw, max(i - 1, 0));
      *b = i ? bs : bj;
      return j + i;
    }
  }
};

// Calls fn(src, at) with each lane's edges e0 + 32 k + lane of a tile of
// 32 * IT edges: their sources src[k] (-1 past the end) and their places at[k]
// in the adjacency.  epos: the sources' first edges (exclusive prefix sums of
// their degrees; EdgeWindow), foff: their lists' starts.  A tile's first
// source comes from a search.  No shared memory and no block barriers: staging
// tiles of 1024 edges through shared memory, with a binary search per edge,
// had the bulk push wait on barriers and shared memory half of the time.
template <int IT, class Fn>
__device__ inline void warp_edges(const int64_t* epos, const int64_t* foff, int64_t nf, int64_t E,
                                  int64_t warp, int64_t nwarps, Fn&& fn) {
  const int lane = threadIdx.x & 31;
  for (int64_t e0 = warp * 32 * IT; e0 < E; e0 += nwarps * 32 * IT) {
    EdgeWindow W(
        max((int64_t)0, warp_upper_bound(epos, nf, e0) - 1), nf,
        [&](int64_t i) { return epos[i]; }, [&](int64_t i) { return foff[i] - epos[i]; });
    int32_t src[IT];
    int64_t at[IT];
#pragma unroll
    for (int k = 0; k < IT; k++) {
      const int64_t eb = e0 + 32 * k;
      int64_t b = 0;
      const int64_t i = W.find(eb, &b);
      src[k] = eb + lane < E ? (int32_t)i : -1;
      at[k] = b + eb + lane;
    }
    fn(src, at);
  }
}

// ---------------------------------------------------------------------------
// Hot destinations.  Adds to one address are served one after another, about
// 2.9 ns an FP64 add, and those to one line nearly so: a Nibble round that
// pushes 7.2M edges of a scale-22 R-MAT graph adds 45,583 of them to its hub
// and 177,000 to its 32 highest-degree vertices, most of those in one or two
// lines; it took 131 us for that.  The adds to the graph's kHot vertices of
// highest degree are summed by their warp, lane h owning vertex h, then by the
// block, and reach memory once per block.  A 256-entry table in shared memory
// (one entry per vertex, no collisions) tells them.
// ---------------------------------------------------------------------------
struct HotShared {
  int2 tab[kHotTab];  // vertex, index
};

// Every thread of the block calls it before the first hot_take.
__device__ inline void hot_load(const HotSet& H, HotShared& M) {
  if (!H.tab) return;
  for (int i = threadIdx.x; i < kHotTab; i += blockDim.x) M.tab[i] = H.tab[i];
  __syncthreads();
}

template <class Sum>
struct HotLane {
  Sum a = {};
  bool any = false;
};

// The edges with a hot w leave their x to the owner's add(sum, x) and become
// w = -1 (all lanes call it).
template <int IT, class Sum, class X, class Bcast, class Add>
__device__ inline void hot_take(const HotSet& H, const HotShared& M, HotLane<Sum>& S,
                                int32_t (&w)[IT], const X (&x)[IT], Bcast&& bcast, Add&& add) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < IT; k++) {
    const int2 e = M.tab[(uint32_t)w[k] * H.mult >> (32 - kHotBits)];
    const bool hit = w[k] >= 0 && e.x == w[k];
    for (unsigned m = __ballot_sync(0xffffffffu, hit); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const X y = bcast(x[k], l);
      if (__shfl_sync(0xffffffffu, e.y, l) == lane) {
        add(S.a, y);
        S.any = true;
      }
    }
    if (hit) w[k] = -1;
  }
}
template <int IT>
__device__ inline void hot_take(const HotSet& H, const HotShared& M, HotLane<double>& S,
                                int32_t (&w)[IT], const double (&sh)[IT]) {
  hot_take(
      H, M, S, w, sh, [](double x, int l) { return __shfl_sync(0xffffffffu, x, l); },
      [](double& a, double x) { a = a + x; });
}

// Every thread of the block calls it; thread h calls done(vertex, sum) for
// each hot vertex met, its warps' sums joined by add.
template <int WARPS, class Sum, class Add, class Done>
__device__ inline void hot_flush(const HotSet& H, const HotLane<Sum>& S, Add&& add, Done&& done) {
  __shared__ Sum s_hot[WARPS][kHot];
  __shared__ unsigned s_any[WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (!__syncthreads_or(S.any)) return;
  const unsigned any = __ballot_sync(0xffffffffu, S.any);
  s_hot[warp][lane] = S.a;
  if (lane == 0) s_any[warp] = any;
  __syncthreads();
  if (warp != 0) return;
  Sum t = {};
  bool met = false;
  for (int k = 0; k < WARPS; k++)
    if ((s_any[k] >> lane) & 1u) {
      add(t, s_hot[k][lane]);
      met = true;
    }
  if (met) done(H.ids[lane], t);
}

}  // namespace lgc
