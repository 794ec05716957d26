// Synchronous frontier diffusions: PR-Nibble (Sec. 3.3), Nibble (Sec. 3.2)
// and HK-PR (Sec. 3.4).
//
// One round = vertexMap over the frontier F (per-algorithm kernel: reads the
// frontier values, updates the vertex's own entries, computes the share it
// sends along each edge) followed by an edgeMap (generic: adds the share to
// the destination's entry of a hash table) and the filter that forms the
// next frontier.
//
// Atomic mode: the edgeMap adds with atomicAdd (the paper's fetchAdd).  The
// next frontier is formed during the edgeMap itself: the one add that takes
// a destination from below its threshold c*d(w) to at least it appends w
// (values only grow, so exactly one add crosses).  Only F and N(F) can
// change, so this equals the paper's filter over the whole sparse set.
//
// Deterministic mode: the edgeMap emits one (destination, share) record per
// edge in frontier order (the frontier is kept in ascending id), sorts the
// records stably by destination, and folds each destination's run left to
// right starting from the value it holds after the vertexMap.  That is the
// order a sequential loop over ascending sources produces, so p, r and every
// frontier are bit-identical to it.  The filter then compacts the runs whose
// result reaches the threshold; runs are in ascending id, so the next
// frontier is too.
//
// All arithmetic is IEEE binary64 with FMA contraction disabled (--fmad=false),
// each expression evaluated in the order written.
#include <math.h>

#include <algorithm>
#include <type_traits>
#include <vector>
#include <string.h>

#include "common.cuh"
#include "edges.cuh"
#include "foldwarp.cuh"
#include "fp64lite.cuh"
#include "fx128.cuh"
#include "lookback.cuh"
#include "prim.cuh"
#include "rounds.cuh"

namespace lgc {

namespace {

constexpr int kEdgeItems = 4;
constexpr int kEdgeTile = kBlock * kEdgeItems;  // edges per block and pass

enum FrontierMode { kFmNone = 0, kFmThreshold = 1, kFmInserted = 2 };

// Adds every thread's count n into *counter with one atomic per block (a
// per-warp atomic on one address queues when a launch has many warps).  All
// threads of the block call it, once, where every thread arrives.
__device__ inline void flush_count(int64_t n, int64_t* counter) {
  __shared__ int64_t s_cnt[kBlock / 32];
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  if ((threadIdx.x & 31) == 0) s_cnt[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t t = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); k++) t += s_cnt[k];
    if (t) atomicAdd((unsigned long long*)counter, (unsigned long long)t);
  }
}

__device__ inline void count_inserted(int ins, int64_t* counter) {
  const unsigned active = __activemask();
  const unsigned m = __ballot_sync(active, ins);
  if (m && (threadIdx.x & 31) == __ffs(active) - 1)
    atomicAdd((unsigned long long*)counter, (unsigned long long)__popc(m));
}

// ---------------------------------------------------------------------------
// vertexMap kernels.  Each writes, per frontier entry i: share[i], the
// record count cnt[i] (d(v), plus one self record in deterministic mode when
// the vertex itself is a key of the destination table) and foff[i] = off[v].
// ---------------------------------------------------------------------------

// PR-Nibble, Fig. alg:pr-nibble (rule 1) / alg:pr-nibble2 (rule 0).  T holds
// r in slot.val and p in T.p[slot]; r' is updated in place (every read of r
// in the round is of a frontier vertex, done here before the edgeMap).
__global__ void vmap_prnibble_kernel(int64_t nf, const int32_t* __restrict__ fv,
                                     const int32_t* __restrict__ fs, Table T,
                                     const int64_t* __restrict__ off, double alpha, double cs,
                                     double cn, double eps, int rule, int det, int self_append,
                                     double* __restrict__ share, int64_t* __restrict__ cnt,
                                     int64_t* __restrict__ foff, int32_t* nfv, int32_t* nfs,
                                     int32_t ncap, Counters* C) {
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nf;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = base + threadIdx.x;
    bool pred = false;
    int32_t v = 0, s = 0;
    int64_t d = 0;
    if (i < nf) {
      v = fv[i];
      s = fs[i];
      const bool ok = s >= 0;  // always true unless a table overflowed (flagged)
      const double r = ok ? *tb_val(T, s) : 0.0;
      const int64_t o0 = off[v];
      d = off[v + 1] - o0;
      double sh, rbase;
      if (rule == 0) {
        if (ok) T.p[s] = T.p[s] + cs * r;
        rbase = 0.0;
        sh = (cn * r) / (double)d;
      } else {
        if (ok) T.p[s] = T.p[s] + alpha * r;
        rbase = ((1.0 - alpha) * r) / 2.0;
        sh = ((1.0 - alpha) * r) / (2.0 * (double)d);
      }
      if (ok) *tb_val(T, s) = rbase;
      share[i] = sh;
      cnt[i] = d + (det ? 1 : 0);
      foff[i] = o0;
      pred = ok && self_append && rule == 1 && rbase >= eps * (double)d;
    }
    frontier_append(pred, v, s, d, nfv, nfs, C, ncap);
  }
}

// Nibble, Fig. alg:nibble: p'[v] = p[v]/2 on the frontier (S = p, D = p',
// fresh), share p[v]/(2 d(v)).
__global__ void vmap_nibble_kernel(int64_t nf, const int32_t* __restrict__ fv,
                                   const int32_t* __restrict__ fs, Table S, Table D,
                                   const int64_t* __restrict__ off, double eps, int fmode,
                                   int det, int self_append, double* __restrict__ share,
                                   int64_t* __restrict__ cnt,
                                   int64_t* __restrict__ foff, int32_t* nfv, int32_t* nfs,
                                   int32_t ncap, Counters* C) {
  int64_t nins = 0;  // counted once per block
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nf;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = base + threadIdx.x;
    bool pred = false;
    int ins = 0;
    int32_t v = 0, ds = 0;
    int64_t d = 0;
    if (i < nf) {
      v = fv[i];
      const double pv = fs[i] >= 0 ? *tb_val(S, fs[i]) : 0.0;
      const int64_t o0 = off[v];
      d = off[v + 1] - o0;
      ds = (int32_t)tb_find_or_insert(D, v, &ins, &C->err);
      const double self = pv / 2.0;
      if (ds >= 0) *tb_val(D, ds) = self;
      share[i] = pv / (2.0 * (double)d);
      cnt[i] = d + (det ? 1 : 0);
      foff[i] = o0;
      if (self_append && ds >= 0)
        pred = fmode == kFmInserted ? true : self >= eps * (double)d;
    }
    nins += ins;
    frontier_append(pred, v, ds, d, nfv, nfs, C, ncap);
  }
  flush_count(nins, &C->aux);
}

// HK-PR, Fig. alg:hkpr: p[v] += r[v] on the frontier; share
// t r[v]/((j+1) d(v)) or, on the last level, r[v]/d(v).
__global__ void vmap_hkpr_kernel(int64_t nf, const int32_t* __restrict__ fv,
                                 const int32_t* __restrict__ fs, Table S, Table P,
                                 const int64_t* __restrict__ off, double t, int j, int last,
                                 double* __restrict__ share, int64_t* __restrict__ cnt,
                                 int64_t* __restrict__ foff, Counters* C) {
  int64_t nins = 0;  // counted once per block
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nf;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = base + threadIdx.x;
    int ins = 0;
    if (i < nf) {
      const int32_t v = fv[i];
      const double r = fs[i] >= 0 ? *tb_val(S, fs[i]) : 0.0;
      const int64_t o0 = off[v];
      const int64_t d = off[v + 1] - o0;
      const int64_t ps = tb_find_or_insert(P, v, &ins, &C->err);
      if (ps >= 0) *tb_val(P, ps) = *tb_val(P, ps) + r;
      share[i] = last ? r / (double)d : (t * r) / ((double)(j + 1) * (double)d);
      cnt[i] = d;
      foff[i] = o0;
    }
    nins += ins;
  }
  flush_count(nins, &C->aux);
}

// ---------------------------------------------------------------------------
// edgeMap, atomic mode, edge-balanced over warps (edges.cuh).  Each thread
// takes kEdgeItems edges through the phases side by side: all columns, first
// probes, slots, adds and crossings.  Consecutive threads read consecutive
// col[] entries.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kBlock)
    emap_atomic_kernel(const int32_t* __restrict__ col, const int32_t* __restrict__ deg,
                       const double* __restrict__ share, const int64_t* __restrict__ epos,
                       const int64_t* __restrict__ foff, int64_t nf, int64_t E_host,
                       const int64_t* __restrict__ E_dev, HotSet H, Table D, double c, int fmode,
                       int32_t* nfv, int32_t* nfs, int32_t ncap, Counters* C) {
  __shared__ HotShared s_tab;
  HotLane<double> S;
  hot_load(H, s_tab);
  // the device-computed total bounds every edge index, whatever the host passed
  const int64_t E = min(E_host, *E_dev);
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t nins = 0;  // counted once per block
  warp_edges<kEdgeItems>(epos, foff, nf, E, warp, nwarps, [&](const int32_t* src,
                                                              const int64_t* at) {
    int32_t w[kEdgeItems];
    double sh[kEdgeItems];
#pragma unroll
    for (int k = 0; k < kEdgeItems; k++) {
      w[k] = -1;
      sh[k] = 0.0;
      if (src[k] >= 0) {
        w[k] = col[at[k]];
        sh[k] = share[src[k]];
      }
    }
    if (H.tab) hot_take(H, s_tab, S, w, sh);
    // Resolve every item's slot before any atomic, so the first-probe loads
    // (or bitmap loads) of all items are in flight together.
    int32_t slot[kEdgeItems];
    int ins[kEdgeItems];
    uint32_t probe[kEdgeItems];
#pragma unroll
    for (int k = 0; k < kEdgeItems; k++) {
      ins[k] = 0;
      probe[k] = 0;
      if (w[k] >= 0)
        probe[k] = D.dense ? __ldcg(&D.bits[w[k] >> 5])
                           : (uint32_t)__ldcg(&D.s[hash_slot(w[k], D.shift)].key);
    }
#pragma unroll
    for (int k = 0; k < kEdgeItems; k++) {
      slot[k] = -1;
      if (w[k] < 0) continue;
      if (D.dense) {
        slot[k] = w[k];
        const uint32_t m = 1u << (w[k] & 31);
        if (!(probe[k] & m) && !(atomicOr(&D.bits[w[k] >> 5], m) & m)) ins[k] = 1;
      } else if ((int32_t)probe[k] == w[k] + 1) {
        slot[k] = (int32_t)hash_slot(w[k], D.shift);
      } else {
        slot[k] = (int32_t)ht_find_or_insert(D, w[k], &ins[k], &C->err);
      }
    }
    // All adds issued back to back; their returned old values decide the
    // threshold crossings.
    double old[kEdgeItems];
#pragma unroll
    for (int k = 0; k < kEdgeItems; k++)
      old[k] = slot[k] >= 0 ? atomicAdd(tb_val(D, slot[k]), sh[k]) : 0.0;
    bool pred[kEdgeItems];
    int64_t dw[kEdgeItems];
#pragma unroll
    for (int k = 0; k < kEdgeItems; k++) {
      pred[k] = false;
      dw[k] = 0;
      if (slot[k] < 0) continue;
      if (fmode == kFmThreshold) {
        const double nv = old[k] + sh[k];
        if (nv >= c) {  // c*d(w) >= c for d(w) >= 1: cheap pre-test
          dw[k] = deg[w[k]];
          const double thr = c * (double)dw[k];
          pred[k] = old[k] < thr && nv >= thr;
        }
      } else if (fmode == kFmInserted && ins[k]) {
        dw[k] = deg[w[k]];
        pred[k] = true;
      }
    }
#pragma unroll
    for (int k = 0; k < kEdgeItems; k++) {
      nins += ins[k];
      frontier_append(pred[k], w[k], slot[k], dw[k], nfv, nfs, C, ncap);
    }
  });
  // the hot vertices' sums, each as one add: the one that takes the vertex
  // across its threshold appends it
  const auto join = [](double& a, double x) { a = a + x; };
  hot_flush<kBlock / 32>(H, S, join, [&](int32_t w, double sh) {
    int ins = 0;
    const int64_t s = tb_find_or_insert(D, w, &ins, &C->err);
    if (s < 0) return;
    nins += ins;
    const double old = atomicAdd(tb_val(D, s), sh);
    const int64_t d = deg[w];
    const double thr = c * (double)d;
    const bool pred = fmode == kFmThreshold ? old < thr && old + sh >= thr
                                            : fmode == kFmInserted && ins != 0;
    if (!pred) return;
    const int32_t pos = atomicAdd(&C->next_size, 1);
    atomicAdd((unsigned long long*)&C->next_edges, (unsigned long long)d);
    if (pos < ncap) {
      nfv[pos] = w;
      nfs[pos] = (int32_t)s;
    } else {
      atomicOr(&C->err, kErrFrontierOverflow);
    }
  });
  flush_count(nins, &C->inserted);
}

// ---------------------------------------------------------------------------
// edgeMap for bulk rounds (atomic mode, dense destination): the adds are
// fire-and-forget reductions (no returned value, so nothing waits on them)
// and the key is marked in the presence bitmap; the next frontier is formed
// afterwards by the dense filter.  Also used for the last HK-PR level (no
// frontier) in either table form.
// ---------------------------------------------------------------------------
constexpr int kRedItems = 8;

__global__ void __launch_bounds__(kBlock)
    emap_red_kernel(const int32_t* __restrict__ col, const double* __restrict__ share,
                    const int64_t* __restrict__ epos, const int64_t* __restrict__ foff,
                    int64_t nf, int64_t E_host, const int64_t* __restrict__ E_dev, HotSet H,
                    Table D, int mark, Counters* C) {
  __shared__ HotShared s_tab;
  HotLane<double> S;
  hot_load(H, s_tab);
  const int64_t E = min(E_host, *E_dev);
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t nins = 0;  // counted once per block
  warp_edges<kRedItems>(epos, foff, nf, E, warp, nwarps, [&](const int32_t* src,
                                                             const int64_t* at) {
    int32_t w[kRedItems];
    double sh[kRedItems];
#pragma unroll
    for (int k = 0; k < kRedItems; k++) {
      w[k] = -1;
      sh[k] = 0.0;
      if (src[k] >= 0) {
        w[k] = col[at[k]];
        sh[k] = share[src[k]];
      }
    }
    if (H.tab) hot_take(H, s_tab, S, w, sh);
    if (D.dense) {
      // nothing waits for a result here: the adds are reductions, and the keys
      // they create are marked by the filter pass that follows (DenseQualWord)
      // or, without one (mark) or where the share is zero, by another reduction
      // unless they are marked already
#pragma unroll
      for (int k = 0; k < kRedItems; k++)
        if (w[k] >= 0) atomicAdd(&D.dval[w[k]], sh[k]);
#pragma unroll
      for (int k = 0; k < kRedItems; k++) {
        if (w[k] < 0 || (!mark && sh[k] > 0.0)) continue;
        const uint32_t m = 1u << (w[k] & 31);
        if (!(__ldcg(&D.bits[w[k] >> 5]) & m)) nins += !(atomicOr(&D.bits[w[k] >> 5], m) & m);
      }
    } else {
#pragma unroll
      for (int k = 0; k < kRedItems; k++) {
        if (w[k] < 0) continue;
        int ins = 0;
        const int64_t s = ht_find_or_insert(D, w[k], &ins, &C->err);
        if (s >= 0) atomicAdd(&D.s[s].val, sh[k]);
        nins += ins;
      }
    }
  });
  const auto join = [](double& a, double x) { a = a + x; };
  hot_flush<kBlock / 32>(H, S, join, [&](int32_t w, double sh) {
    int ins = 0;
    const int64_t s = tb_find_or_insert(D, w, &ins, &C->err);
    if (s >= 0) atomicAdd(tb_val(D, s), sh);
    nins += ins;
  });
  flush_count(nins, &C->inserted);
}

// Sources without edges (lgc_graph::sinks) behind the others, starting where
// the edges end (EdgeWindow).  has[i]: cnt[i] > 0; pos: its exclusive prefix
// sums, *npos in all.
__global__ void has_edges_kernel(const int64_t* __restrict__ cnt, int64_t nf,
                                 int64_t* __restrict__ has) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf;
       i += (int64_t)gridDim.x * blockDim.x)
    has[i] = cnt[i] > 0;
}
__global__ void sinks_last_kernel(int64_t nf, const int64_t* __restrict__ cnt,
                                  const int64_t* __restrict__ pos,
                                  const int64_t* __restrict__ npos,
                                  const int64_t* __restrict__ E_dev,
                                  const double* __restrict__ share,
                                  const int64_t* __restrict__ epos,
                                  const int64_t* __restrict__ foff, double* __restrict__ share_out,
                                  int64_t* __restrict__ epos_out, int64_t* __restrict__ foff_out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf;
       i += (int64_t)gridDim.x * blockDim.x) {
    const bool any = cnt[i] > 0;
    const int64_t at = any ? pos[i] : *npos + i - pos[i];
    share_out[at] = share[i];
    epos_out[at] = any ? epos[i] : *E_dev;
    foff_out[at] = foff[i];
  }
}

// Filter of a dense set after a bulk push, in ascending vertex order.  The
// push leaves the presence bits of the keys it created to this pass, which
// reads the values anyway: a vertex with a value that is not zero is a key
// (the push marks the destinations of zero shares itself).  Vertex v qualifies
// when it is a key and its value reaches c*d(v) (kFmThreshold) or always
// (kFmInserted); the qualifying vertices are compacted (words_compact), their
// degrees summed, and the new keys counted.
struct DenseQualWord {
  Table D;
  const int32_t* deg;
  int64_t n;
  LiteThr c;
  int fmode;
  int64_t* inserted;
  __device__ void marked(int k) const {
    atomicAdd((unsigned long long*)inserted, (unsigned long long)k);
  }
  __device__ uint32_t operator()(int64_t w, bool in, int* fresh) const {
    const int lane = threadIdx.x & 31;
    const int64_t wb = w - lane;
    const uint32_t m = in ? D.bits[w] : 0u;
    double x[kCmpWarpWords];
#pragma unroll
    for (int j = 0; j < kCmpWarpWords; j++) {
      const int64_t v = (wb + j) * 32 + lane;
      x[j] = v < n ? D.dval[v] : 0.0;
    }
    uint32_t q = 0;
#pragma unroll
    for (int j = 0; j < kCmpWarpWords; j++) {
      const int64_t v = (wb + j) * 32 + lane;
      const uint32_t mj = __shfl_sync(0xffffffffu, m, j);
      const bool nz = __double_as_longlong(x[j]) != 0;  // no value is -0.0
      const uint32_t key = mj | __ballot_sync(0xffffffffu, nz);
      const uint32_t b = fmode == kFmThreshold
                             ? __ballot_sync(0xffffffffu, nz && lite_reaches(x[j], c, deg[v]))
                             : key;
      if (lane == j) {
        q = b;
        if (key != m) {
          D.bits[w] = key;
          *fresh = __popc(key & ~m);
        }
      }
    }
    return q;
  }
};

// ---------------------------------------------------------------------------
// Pull edgeMap (deterministic mode, dense rounds).  Instead of scattering
// from the frontier, every vertex w gathers from its neighbours that are in
// the frontier.  Adjacency lists are sorted, so w meets its in-frontier
// neighbours in ascending id: folding their shares left to right from w's
// current value is exactly the canonical order, with no records and no sort.
// The frontier is given as one double per vertex, sh[v]: +0.0 (all bits
// zero) for a vertex outside the frontier, its share for a frontier vertex,
// and -0.0 for a frontier vertex whose share is zero.  So one gather gives
// both membership (any bit set) and the value, and adding a member's -0.0 to
// a non-negative value changes nothing, exactly as its +0.0 share would.
// Vertices of degree <= kPullLight use one thread, the rest (ascending list
// g->heavy) are read in batches by warps.  Qualifying vertices are marked in
// qbits for an ordered compaction.
// ---------------------------------------------------------------------------
__device__ inline bool pull_member(double s) { return __double_as_longlong(s) != 0; }

__global__ void pull_scatter_kernel(int64_t nf, const int32_t* __restrict__ fv,
                                    const double* __restrict__ share, double* __restrict__ sh,
                                    int clear) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = fv[i];
    if (clear) {
      sh[v] = 0.0;
      continue;
    }
    const double x = share[i];
    sh[v] = pull_member(x) ? x : -0.0;
  }
}

__device__ inline bool pull_qualifies(double acc, int64_t d, LiteThr c, int fmode) {
  if (fmode == kFmThreshold) return lite_reaches(acc, c, (int32_t)d);
  return fmode == kFmInserted;
}

// Deterministic pull, vertices of degree 1..kPullLight: one thread folds its
// list in order (acc <- RN(acc + s) from the present value), taking the
// vertices from the graph's list grouped by degree so that a warp's chains
// have one length.  qbits is cleared before; qualifying vertices are ORed in.
__global__ void pull_light_kernel(LightView V, const double* __restrict__ sh, Table D, LiteThr c,
                                  int fmode, uint32_t* __restrict__ qbits, Counters* C) {
  const int stride = V.stride();
  int64_t nins = 0;  // keys inserted here, counted once per block
  for (int64_t i = V.first() + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V.end;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i < V.beg) continue;
    const LightItem it = V.items[i];
    const int32_t* col = V.columns(i, it);
    const int32_t w = it.w;
    const uint32_t m = 1u << (w & 31);
    const bool present = (D.bits[w >> 5] & m) != 0;
    double acc = present ? D.dval[w] : 0.0;
    bool touched = present;
    for (int k = 0; k < it.d; k++) {
      const double x = sh[col[k * stride]];
      if (pull_member(x)) {
        acc = acc + x;
        touched = true;
      }
    }
    if (touched) {
      D.dval[w] = acc;
      if (!present && !(atomicOr(&D.bits[w >> 5], m) & m)) nins++;
      if (pull_qualifies(acc, it.d, c, fmode)) atomicOr(&qbits[w >> 5], m);
    }
  }
  flush_count(nins, &C->inserted);
}

// Heavy vertices are read in batches of 32 * BATCH edges: every lane issues
// the loads of BATCH edges (column, then share) before any of them is used,
// so one batch costs two memory round trips; BATCH is the graph's tuned value
// (kPullBatch until tuned).
constexpr int kPullBatch = 8;

// Writes a heavy vertex's gathered value (lane 0 calls it); 1 if the vertex
// became a key here (the caller counts it).
__device__ inline int pull_finish(const Table& D, int32_t w, int64_t d, double acc, bool touched,
                                  bool present, LiteThr c, int fmode, uint32_t* qbits) {
  if (!touched) return 0;
  const uint32_t m = 1u << (w & 31);
  D.dval[w] = acc;
  const int ins = !present && !(atomicOr(&D.bits[w >> 5], m) & m);
  if (pull_qualifies(acc, d, c, fmode)) atomicOr(&qbits[w >> 5], m);
  return ins;
}

// Deterministic mode, vertices of degree (kPullLight, kDetBig]: one lane per
// vertex folds its in-frontier shares in adjacency order with FP64 adds --
// the fold's definition, so bit-identical by construction (a vertex outside
// the frontier has the share +0.0, which adds nothing to a value of at least
// +0.0).  The vertices are taken longest list first and a warp's lanes have
// lists of similar length, so every add is issued for (nearly) all 32 lanes.
//
// A quarter of an SM takes an FP64 warp instruction every 64 cycles, dependent
// or not, so two warps a quarter keep its pipe busy, and what matters is that
// the longest lists lie one to a quarter: a block an SM, its warps' first
// slices dealt across the blocks (longest first), the others taken as warps
// come free.  A batch's shares and the next one's columns are read before the
// adds of the batch before.  The 15.1M edges of a scale-20 R-MAT graph's middle
// lists: 137 us with neighbouring slices in one block, 104 dealt to two blocks
// of 8 warps an SM, 88 so; 94 with 12 warps, 96 with 16, 111 with 24 and
// batches of 8; 195 with the shares copied ahead to shared memory.  Of it 60
// are the adds and 75 the loads, each by itself.
constexpr int kMidB = 16;

__global__ void __launch_bounds__(kBlock, 1)
    pull_mid_det_kernel(LightView V, const double* __restrict__ sh, Table D, LiteThr c, int fmode,
                        uint32_t* __restrict__ qbits, unsigned* __restrict__ ticket, Counters* C) {
  const int lane = threadIdx.x & 31;
  const int stride = V.stride();
  int64_t nins = 0;  // keys inserted here
  unsigned t = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  for (bool own = true;; own = false) {
    if (!own) {
      if (lane == 0) t = gridDim.x * (kBlock / 32) + atomicAdd(ticket, 1u);
      t = __shfl_sync(0xffffffffu, t, 0);
    }
    const int64_t base = V.first() + 32 * (int64_t)t;
    if (base >= V.end) break;
    const int64_t i = base + lane;
    if (i < V.beg || i >= V.end) continue;
    const LightItem it = V.items[i];
    const int32_t* __restrict__ col = V.columns(i, it);
    const int32_t w = it.w, d = it.d;
    const uint32_t m = 1u << (w & 31);
    const bool present = (D.bits[w >> 5] & m) != 0;
    double acc = present ? D.dval[w] : 0.0;
    uint64_t any = 0;
    int32_t u[kMidB];
    double x[kMidB];
    auto columns = [&](int k) {
#pragma unroll
      for (int j = 0; j < kMidB; j++) u[j] = k + j < d ? col[(k + j) * stride] : -1;
    };
    columns(0);
#pragma unroll
    for (int j = 0; j < kMidB; j++) x[j] = u[j] >= 0 ? sh[u[j]] : 0.0;
    columns(kMidB);
    for (int k = 0; k < d; k += kMidB) {
      double xn[kMidB];
#pragma unroll
      for (int j = 0; j < kMidB; j++) xn[j] = u[j] >= 0 ? sh[u[j]] : 0.0;
      columns(k + 2 * kMidB);
#pragma unroll
      for (int j = 0; j < kMidB; j++) {  // in order: j ascending is adjacency order
        acc = acc + x[j];
        any |= (uint64_t)__double_as_longlong(x[j]);
      }
#pragma unroll
      for (int j = 0; j < kMidB; j++) x[j] = xn[j];
    }
    if (present || any) {
      D.dval[w] = acc;
      if (!present && !(atomicOr(&D.bits[w >> 5], m) & m)) nins++;
      if (pull_qualifies(acc, d, c, fmode)) atomicOr(&qbits[w >> 5], m);
    }
  }
  flush_count(nins, &C->inserted);
}

// ---------------------------------------------------------------------------
// Deterministic mode, vertices of degree > kDetBig: the fold of the whole
// list is split into 256-edge segments that are worked on in parallel.
//  1. det_seg_sum: each segment's sum to about 20 bits and whether it holds a
//     member; the gathered shares are kept for 3 and 4 (up to kDetKeep
//     segments, beyond which those gather again).
//  2. det_seg_predict: per vertex, a running sum of the segment sums
//     predicts the binade the fold is in at each segment's start (the
//     prediction misses only next to a power of two).
//  3. det_seg_step: each segment's composed integer step (see fold_step) for
//     its predicted binade.
//  4. det_seg_verify: one warp per vertex walks its segments in order, up to
//     32 at a time: while the fold's actual binade is the predicted one and
//     the steps composed so far keep the value below 2^53, they are the exact
//     fold of their segments (the value only grows, so no intermediate value
//     left the binade); the segment that does not is folded element by
//     element (fold_batch), its shares loaded ahead where the next one's
//     prediction tells it.
// The result is the sequential fold, bit for bit.
// ---------------------------------------------------------------------------
// A sum for prediction only: the shares' leading 21 bits in units of the
// largest one's last, in 32-bit integers (256 of them stay below 2^29).  The
// plain sum's 13 FP64 adds a segment were the pass's bound.
__global__ void det_seg_sum_kernel(const int32_t* __restrict__ col,
                                   const DetSeg* __restrict__ segs, int64_t nsegs,
                                   const double* __restrict__ sh, double* __restrict__ segsum,
                                   int32_t* __restrict__ segany, double* __restrict__ kept) {
  const int lane = threadIdx.x & 31;
  const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = warp0; k < nsegs; k += nwarps) {
    const DetSeg S = segs[k];
    int32_t u[8];
#pragma unroll
    for (int j = 0; j < 8; j++) u[j] = 32 * j + lane < S.len ? col[S.beg + 32 * j + lane] : -1;
    double v[8];
#pragma unroll
    for (int j = 0; j < 8; j++) v[j] = u[j] >= 0 ? sh[u[j]] : 0.0;
    uint32_t top = 0;
    bool mem = false;
#pragma unroll
    for (int j = 0; j < 8; j++) {
      if (kept) kept[kDetSeg * k + 32 * j + lane] = v[j];
      mem = mem || pull_member(v[j]);
      top = max(top, (uint32_t)__double2hiint(v[j]) >> 20 & 2047u);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    uint32_t x = 0;
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const uint32_t hi = (uint32_t)__double2hiint(v[j]);
      const uint32_t be = hi >> 20 & 2047u;
      if (be) x += ((hi & 0xFFFFFu) | 0x100000u) >> min(top - be, 31u);
    }
    x = __reduce_add_sync(0xffffffffu, x);
    const bool any = __any_sync(0xffffffffu, mem);
    if (lane == 0) {
      // x * 2^(top - 1043); below 2^-1002 predicted as nothing
      segsum[k] = top > 20 ? (double)x * __hiloint2double((int)((top - 20) << 20), 0) : 0.0;
      segany[k] = any ? 1 : 0;
    }
  }
}

__global__ void det_seg_predict_kernel(const int32_t* __restrict__ big_w,
                                       const int64_t* __restrict__ seg0, int64_t nbig, Table D,
                                       const double* __restrict__ segsum,
                                       int32_t* __restrict__ pred) {
  const int lane = threadIdx.x & 31;
  const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = warp0; b < nbig; b += nwarps) {
    const int32_t w = big_w[b];
    const bool present = (D.bits[w >> 5] >> (w & 31)) & 1u;
    double acc = present ? D.dval[w] : 0.0;
    const int64_t k1 = seg0[b + 1];
    for (int64_t k0 = seg0[b]; k0 < k1; k0 += 32) {
      const int64_t k = k0 + lane;
      double x = k < k1 ? segsum[k] : 0.0;
      for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      double before = __shfl_up_sync(0xffffffffu, x, 1);
      if (lane == 0) before = 0.0;
      if (k < k1) pred[k] = fold_binade(acc + before);
      acc += __shfl_sync(0xffffffffu, x, 31);
    }
  }
}

// Lane l's eight shares of segment k (positions 8 l .. 8 l + 7).
__device__ inline void det_seg_shares(const double* __restrict__ kept,
                                      const int32_t* __restrict__ col,
                                      const DetSeg* __restrict__ segs,
                                      const double* __restrict__ sh, int64_t k, int lane,
                                      double (&v)[8]) {
  if (kept) {
    const double2* p = reinterpret_cast<const double2*>(kept + kDetSeg * k + 8 * lane);
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const double2 x = p[q];
      v[2 * q] = x.x;
      v[2 * q + 1] = x.y;
    }
    return;
  }
  const DetSeg S = segs[k];
  int32_t u[8];
#pragma unroll
  for (int q = 0; q < 8; q++) u[q] = 8 * lane + q < S.len ? col[S.beg + 8 * lane + q] : -1;
#pragma unroll
  for (int q = 0; q < 8; q++) v[q] = u[q] >= 0 ? sh[u[q]] : 0.0;
}

__global__ void det_seg_step_kernel(const int32_t* __restrict__ col,
                                    const DetSeg* __restrict__ segs, int64_t nsegs,
                                    const double* __restrict__ sh,
                                    const double* __restrict__ kept,
                                    const int32_t* __restrict__ pred,
                                    FoldStep* __restrict__ step) {
  const int lane = threadIdx.x & 31;
  const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = warp0; k < nsegs; k += nwarps) {
    const int bu = pred[k];
    double v[8];
    det_seg_shares(kept, col, segs, sh, k, lane, v);
    int64_t x0 = 0, x1 = 1;  // the lane's steps from an even and from an odd value
    bool par = false;
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const FoldNear f = fold_near(v[j], bu);
      x0 = fold_take(f, x0);
      x1 = fold_take(f, x1);
      par = par || f.tie;
    }
    FoldStep F = {x0, x1 - 1};
    if (!__any_sync(0xffffffffu, par)) {  // no ties: plain sums
      for (int o = 16; o > 0; o >>= 1) F.g0 += __shfl_xor_sync(0xffffffffu, F.g0, o);
      F.g1 = F.g0;
    } else {
      // ordered reduction: lane l's steps come before lane l+1's
      for (int o = 1; o < 32; o <<= 1) {
        FoldStep q;
        q.g0 = __shfl_down_sync(0xffffffffu, F.g0, o);
        q.g1 = __shfl_down_sync(0xffffffffu, F.g1, o);
        if ((lane & (2 * o - 1)) == 0) F = fold_compose(F, q);
      }
    }
    // a step past 2^53 is never taken; capped, 32 of them stay in 64 bits
    if (lane == 0) step[k] = {min(F.g0, kFoldBig), min(F.g1, kFoldBig)};
  }
}

__global__ void __launch_bounds__(kBlock, 3)
    det_seg_verify_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                          const DetSeg* __restrict__ segs, const int32_t* __restrict__ big_w,
                          const int64_t* __restrict__ seg0, int64_t nbig,
                          const double* __restrict__ sh, const double* __restrict__ kept,
                          const int32_t* __restrict__ pred, const FoldStep* __restrict__ step,
                          const int32_t* __restrict__ segany, Table D, LiteThr c, int fmode,
                          uint32_t* __restrict__ qbits, Counters* C) {
  const int lane = threadIdx.x & 31;
  // the vertices are longest first: neighbours go to different blocks
  const int64_t warp0 = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t nins = 0;
  for (int64_t b = warp0; b < nbig; b += nwarps) {
    const int32_t w = big_w[b];
    const bool present = (D.bits[w >> 5] >> (w & 31)) & 1u;
    double acc = present ? D.dval[w] : 0.0;  // >= +0, the same in every lane
    bool touched = present;
    const int64_t kb = seg0[b], k1 = seg0[b + 1];
    // 32 segments' predictions and steps, one per lane
    int pn = -1;
    FoldStep sn = {0, 0};
    int an = 0;
    auto fetch = [&](int64_t k) {
      pn = k < k1 ? pred[k] : -1;
      sn = k < k1 ? step[k] : FoldStep{0, 0};
      an = k < k1 ? segany[k] : 0;
    };
    fetch(kb + lane);
    for (int64_t k0 = kb; k0 < k1; k0 += 32) {
      const int pl = pn;
      const FoldStep sl = sn;
      touched = touched || __any_sync(0xffffffffu, an != 0);
      fetch(k0 + 32 + lane);
      const int cnt = (int)min((int64_t)32, k1 - k0);
      // segments after which another binade is predicted: the fold leaves
      // its binade in them; the first one's shares are on their way while
      // those before it are taken
      int after = __shfl_down_sync(0xffffffffu, pl, 1);
      const int next = __shfl_sync(0xffffffffu, pn, 0);
      if (lane == 31) after = next;
      unsigned cross = __ballot_sync(0xffffffffu, lane < cnt && after != pl && after >= 0);
      double v[8];
      int held = -1;  // the segment v belongs to
      auto ahead = [&](int j) {
        cross &= j < 32 ? 0xffffffffu << j : 0u;
        if (cross) {
          held = __ffs(cross) - 1;
          det_seg_shares(kept, col, segs, sh, k0 + held, lane, v);
        }
      };
      ahead(0);
      for (int j = 0; j < cnt;) {
        const int bu = fold_binade(acc);
        // the segments from j on that are predicted in this binade
        const unsigned same = __ballot_sync(0xffffffffu, lane < cnt && pl == bu) >> j;
        const int run = same == 0xffffffffu ? 32 : __ffs(~same) - 1;
        if (run > 0) {
          const bool in = lane >= j && lane < j + run;
          FoldStep P = in ? sl : FoldStep{0, 0};
          if (!__any_sync(0xffffffffu, P.g0 != P.g1)) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int64_t q = __shfl_up_sync(0xffffffffu, P.g0, o);
              if (lane >= o) P.g0 += q;
            }
            P.g1 = P.g0;
          } else {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              FoldStep q;
              q.g0 = __shfl_up_sync(0xffffffffu, P.g0, o);
              q.g1 = __shfl_up_sync(0xffffffffu, P.g1, o);
              if (lane >= o) P = fold_compose(q, P);
            }
          }
          const int64_t A = fold_apply(P, fold_int(acc));
          const unsigned over = __ballot_sync(0xffffffffu, in && A >= kFoldTop);
          const int t = over ? __ffs(over) - 1 : j + run;
          if (t > j) acc = fold_double(__shfl_sync(0xffffffffu, A, t - 1), bu);
          j = t;
          if (j >= cnt) break;
        }
        // the prediction missed or the segment leaves the binade: fold it
        // element by element
        if (held != j) det_seg_shares(kept, col, segs, sh, k0 + j, lane, v);
        if (acc == 0.0) {
          // a fold that starts leaves its binade every few of the first
          // shares, and fold_batch starts again each time: those
          // by FP64 adds (shares 0 .. 31 are in lanes 0 .. 3)
#pragma unroll
          for (int l = 0; l < 4; l++)
#pragma unroll
            for (int q = 0; q < 8; q++) acc = acc + __shfl_sync(0xffffffffu, v[q], l);
          if (lane < 4)
#pragma unroll
            for (int q = 0; q < 8; q++) v[q] = 0.0;
        }
        acc = fold_batch(acc, v, lane);
        j++;
        ahead(j);
      }
    }
    if (lane == 0)
      nins += pull_finish(D, w, off[w + 1] - off[w], acc, touched, present, c, fmode, qbits);
  }
  flush_count(nins, &C->inserted);
}

// ---------------------------------------------------------------------------
// Pull edgeMap, atomic mode.  The order of the adds is free, so the gather
// sums in 128-bit fixed point (fx128.cuh) instead of FP64: per edge one
// 16-byte load and four integer adds, and per vertex one rounding.  The
// round's scale L comes from the range of the frontier's shares:
// range[0] = max over nonzero shares of (2047 - biased exponent),
// range[1] = max biased exponent (both 0 before the round).
// shx[v] = {X, flag} for a frontier vertex v, {0, 0} otherwise.
// ---------------------------------------------------------------------------
// A share's contribution to the range (emin holds 2047 - biased exponent).
__device__ inline void range_take(double x, int& emin, int& emax) {
  const uint64_t b = fx_bits(x) & kFxMask;
  if (b) {
    const int be = fx_bexp(b);
    emin = max(emin, 2047 - be);
    emax = max(emax, be);
  }
}

// The block's range into range[] (every thread of the block calls it).
__device__ inline void range_flush(int emin, int emax, int32_t* __restrict__ range) {
  __shared__ int s_r[2][kBlock / 32];
  // one atomic pair per block: same-address atomics serialise in L2
  emin = __reduce_max_sync(0xffffffffu, emin);
  emax = __reduce_max_sync(0xffffffffu, emax);
  const int wib = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    s_r[0][wib] = emin;
    s_r[1][wib] = emax;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    emin = threadIdx.x < kBlock / 32 ? s_r[0][threadIdx.x] : 0;
    emax = threadIdx.x < kBlock / 32 ? s_r[1][threadIdx.x] : 0;
    emin = __reduce_max_sync(0xffffffffu, emin);
    emax = __reduce_max_sync(0xffffffffu, emax);
    if (threadIdx.x == 0 && (emin | emax)) {
      atomicMax(&range[0], emin);
      atomicMax(&range[1], emax);
    }
  }
}

__global__ void share_range_kernel(int64_t nf, const double* __restrict__ share,
                                   int32_t* __restrict__ range) {
  int emin = 0, emax = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf;
       i += (int64_t)gridDim.x * blockDim.x)
    range_take(share[i], emin, emax);
  range_flush(emin, emax, range);
}

// HK-PR vertexMap of a pull round gathering 8-byte shares: the step of
// vmap_hkpr_kernel, with the share written straight into the per-vertex
// array the gathers read (pull_scatter_kernel's membership encoding) and, in
// atomic mode (range non-null, zeroed before), the shares' exponent range
// reduced here; a pull round needs no push records.
// The denominators' reciprocals 1 / (m d) by degree d < tab_n, m = j + 1 (1 on
// the last level), come from recip (recip_level_kernel; null: divide).
__global__ void recip_level_kernel(Recip* __restrict__ recip, int32_t tab_n, double m) {
  for (int32_t d = blockIdx.x * blockDim.x + threadIdx.x; d < tab_n; d += gridDim.x * blockDim.x)
    recip[d] = recip_of(m * (double)max(d, 1));
}

__global__ void vmap_hkpr_pull_kernel(int64_t nf, const int32_t* __restrict__ fv,
                                      const int32_t* __restrict__ fs, Table S, Table P,
                                      const int32_t* __restrict__ deg, double t, int j, int last,
                                      const Recip* __restrict__ recip, int32_t tab_n,
                                      double* __restrict__ sh, int32_t* __restrict__ range,
                                      Counters* C) {
  int emin = 0, emax = 0;
  int64_t nins = 0;  // counted once per block
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nf;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = base + threadIdx.x;
    int ins = 0;
    if (i < nf) {
      const int32_t v = fv[i];
      const double r = fs[i] >= 0 ? *tb_val(S, fs[i]) : 0.0;
      const int64_t d = deg[v];
      const int64_t ps = tb_find_or_insert(P, v, &ins, &C->err);
      if (ps >= 0) *tb_val(P, ps) = *tb_val(P, ps) + r;
      const double a = last ? r : t * r, b = last ? (double)d : (double)(j + 1) * (double)d;
      const double x = d < tab_n ? div_by(a, recip[d], b) : a / b;
      sh[v] = pull_member(x) ? x : -0.0;
      range_take(x, emin, emax);
    }
    nins += ins;
  }
  flush_count(nins, &C->aux);
  if (range) range_flush(emin, emax, range);
}

__device__ inline int round_scale(const int32_t* range, int g) {
  return fx_scale(2047 - range[0], range[1], g);
}

// The gathered frontier share as a fixed-point record: either stored so
// (16 bytes per vertex), or stored as the double share with the membership
// encoding of the deterministic pull (+0.0 outside the frontier, -0.0 for a
// zero share) and converted here (8 bytes per vertex, a few integer
// operations per edge).  Same value either way.
__device__ inline Fx to_fx(const Fx& x, int) { return x; }
__device__ inline Fx to_fx(double s, int L) {
  const uint64_t b = fx_bits(s);
  Fx x = fx_from_bits(b, L);  // -0.0 -> 0
  x.hi |= (uint64_t)(b != 0) << 63;
  return x;
}
template <typename SH>
__device__ inline SH no_share();
template <>
__device__ inline Fx no_share<Fx>() {
  return Fx{0, 0};
}
template <>
__device__ inline double no_share<double>() {
  return 0.0;
}

__global__ void pull_scatter_fx_kernel(int64_t nf, const int32_t* __restrict__ fv,
                                       const double* __restrict__ share, Fx* __restrict__ shx,
                                       const int32_t* __restrict__ range, int g, int clear) {
  const int L = clear ? 0 : round_scale(range, g);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf;
       i += (int64_t)gridDim.x * blockDim.x) {
    Fx x = {0, 0};
    if (!clear) {
      x = fx_from_double(share[i], L);
      x.hi |= kFxFlag;
    }
    shx[fv[i]] = x;
  }
}

// Autotuning input: every vertex in the frontier with share 1 (X = 1 at
// the scale the range {1023, 1023} gives).
template <typename SH>
__global__ void tune_fill_kernel(SH* __restrict__ shx, int64_t n, int32_t* __restrict__ range,
                                 int g) {
  const int L = fx_scale(1023, 1023, g);
  const Fx one = fx_from_double(1.0, L);
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    if constexpr (sizeof(SH) == sizeof(Fx)) {
      shx[v] = Fx{one.lo, one.hi | kFxFlag};
    } else {
      shx[v] = 1.0;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    range[0] = 2047 - 1023;
    range[1] = 1023;
  }
}

// A gathered list's sum: W >= 1, 8-byte shares in W windows (FxWindow); W = 0,
// 16-byte records or 8-byte shares over any range, in 128 bits term by term.
template <int W, typename SH>
struct PullSum {
  FxWindow<W> win;
  uint32_t any = 0;
  __device__ void add(double s, int, uint32_t be0) {
    const uint64_t b = fx_bits(s);
    any |= (uint32_t)b | (uint32_t)(b >> 32);
    win.add(b, be0);
  }
  __device__ Fx total() const { return win.total(); }
  __device__ bool member() const { return any != 0; }
};
template <typename SH>
struct PullSum<0, SH> {
  Fx acc = {0, 0};
  uint64_t flag = 0;
  __device__ void add(const SH& s, int L, uint32_t) {
    const Fx x = to_fx(s, L);
    flag |= x.hi;
    fx_add(acc, x);
  }
  __device__ Fx total() const { return acc; }
  __device__ bool member() const { return (flag & kFxFlag) != 0; }
};

// Calls body<W>() for the windows the round's shares need (the same in every
// thread of the grid).
template <typename SH, class Body>
__device__ inline void pull_windows(const int32_t* range, int L, Body&& body) {
  if constexpr (sizeof(SH) == 8) {
    const int w = fx_windows(2047 - range[0], range[1], L);
    if (w == 1) return body(std::integral_constant<int, 1>());
    if (w == 2) return body(std::integral_constant<int, 2>());
  }
  body(std::integral_constant<int, 0>());
}

// Vertices of degree 1..kPullLight, one thread each, taken from the graph's
// list grouped by degree so that the threads of a warp walk lists of one
// length (in id order most of a warp idled behind its longest list); the
// edges are read four at a time (all column loads, then all share loads).
// The bitmap qbits is cleared before this launch; this kernel and the heavy
// one OR their qualifying vertices in.
template <int W, typename SH>
__device__ inline int64_t pull_light_fx_body(const LightView& V, const SH* __restrict__ shx,
                                             uint32_t be0, int L, const Table& D, LiteThr c,
                                             int fmode, uint32_t* __restrict__ qbits) {
  constexpr int kB = W == 0 ? 4 : 8;  // edges in flight (128-bit sums: registers)
  const int stride = V.stride();
  int64_t nins = 0;  // keys inserted here, counted once per block
  for (int64_t i = V.first() + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < V.end;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i < V.beg) continue;
    const LightItem it = V.items[i];
    const int32_t* __restrict__ col = V.columns(i, it);
    const int32_t w = it.w, d = it.d;
    PullSum<W, SH> sum;
    for (int k = 0; k < d; k += kB) {
      int32_t u[kB];
#pragma unroll
      for (int j = 0; j < kB; j++) u[j] = k + j < d ? col[(k + j) * stride] : -1;
      SH raw[kB];
#pragma unroll
      for (int j = 0; j < kB; j++) raw[j] = u[j] >= 0 ? shx[u[j]] : no_share<SH>();
#pragma unroll
      for (int j = 0; j < kB; j++) sum.add(raw[j], L, be0);
    }
    const uint32_t m = 1u << (w & 31);
    const bool present = (D.bits[w >> 5] & m) != 0;
    if (present || sum.member()) {
      const double v = (present ? D.dval[w] : 0.0) + fx_to_double(sum.total(), L);
      D.dval[w] = v;
      if (!present && !(atomicOr(&D.bits[w >> 5], m) & m)) nins++;
      if (pull_qualifies(v, d, c, fmode)) atomicOr(&qbits[w >> 5], m);
    }
  }
  return nins;
}

// Heavy vertices: one warp per work item (at most kPullItem edges of one
// heavy vertex); lanes sum strided parts, then a butterfly.  The item's
// record and the vertex's current state are loaded first and the latter is
// not waited for until the end, so an item costs three dependent memory
// trips (record, columns, shares).  A vertex with one item is finished at
// once; otherwise the item's sum is added into hacc[h] (two 64-bit atomic
// adds, the low word's carry taken from its returned old value) and the warp
// that completes the vertex's last item finishes it and resets the
// accumulators for the next round.
// GL lanes (8, 16 or 32) work on one item; a warp's 32 / GL groups take
// consecutive items.  The loop over items runs the same number of times in
// every lane of the warp (a group past the end works on nothing), so the
// group-wide shuffles always find all their lanes.
template <int W, int BATCH, int GL, typename SH>
__device__ inline int64_t pull_heavy_fx_body(const int64_t* __restrict__ off,
                                             const int32_t* __restrict__ col,
                                             const PullItem* __restrict__ items, int64_t nitems,
                                             const SH* __restrict__ shx, uint32_t be0, int L,
                                             const Table& D, LiteThr c, int fmode,
                                             uint32_t* __restrict__ qbits, Fx* __restrict__ hacc,
                                             int32_t* __restrict__ hcnt,
                                             int32_t* __restrict__ htouch) {
  constexpr int kGroups = 32 / GL;
  int64_t nins = 0;  // vertices that became keys here
  const int lane = threadIdx.x & 31, gl = lane % GL, gid = lane / GL;
  const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t base = warp0 * kGroups; base < nitems; base += nwarps * kGroups) {
    const int64_t it = base + gid;
    const bool valid = it < nitems;
    PullItem I;
    if (valid) {
      I = items[it];
    } else {
      I.beg = 0;
      I.w = 0;
      I.h = 0;
      I.len = 0;
      I.nparts = 1;
    }
    const int32_t w = I.w;
    // the vertex's state, needed only by the group's first lane at the end
    uint32_t bword = 0;
    double cur = 0.0;
    int64_t d = 0;
    if (gl == 0 && valid) {
      bword = D.bits[w >> 5];
      cur = D.dval[w];
      d = off[w + 1] - off[w];
    }
    PullSum<W, SH> sum;
    for (int k0 = 0; k0 < I.len; k0 += GL * BATCH) {
      int32_t u[BATCH];
#pragma unroll
      for (int j = 0; j < BATCH; j++) {
        const int k = k0 + GL * j + gl;
        u[j] = k < I.len ? col[I.beg + k] : -1;
      }
      SH raw[BATCH];
#pragma unroll
      for (int j = 0; j < BATCH; j++) raw[j] = u[j] >= 0 ? shx[u[j]] : no_share<SH>();
#pragma unroll
      for (int j = 0; j < BATCH; j++) sum.add(raw[j], L, be0);
    }
    Fx part = sum.total();
    uint32_t mem = sum.member() ? 1u : 0u;
    for (int o = GL / 2; o > 0; o >>= 1) {  // within the group
      Fx t;
      t.lo = __shfl_xor_sync(0xffffffffu, part.lo, o);
      t.hi = __shfl_xor_sync(0xffffffffu, part.hi, o);
      fx_add(part, t);
      mem |= __shfl_xor_sync(0xffffffffu, mem, o);
    }
    const bool any = mem != 0;
    if (gl != 0 || !valid) continue;
    const bool present = (bword >> (w & 31)) & 1u;
    if (I.nparts == 1) {
      if (present || any)
        nins += pull_finish(D, w, d, (present ? cur : 0.0) + fx_to_double(part, L), true,
                            present, c, fmode, qbits);
      continue;
    }
    const int32_t h = I.h;
    unsigned long long* acc = reinterpret_cast<unsigned long long*>(&hacc[h]);
    part.hi &= kFxMask;
    if (part.lo | part.hi) {
      const unsigned long long old = atomicAdd(&acc[0], (unsigned long long)part.lo);
      const unsigned long long carry = old + part.lo < old ? 1ull : 0ull;
      atomicAdd(&acc[1], (unsigned long long)part.hi + carry);
    }
    if (any) atomicOr(&htouch[h], 1);
    __threadfence();
    if (atomicAdd(&hcnt[h], 1) == I.nparts - 1) {
      __threadfence();
      Fx total;
      total.lo = atomicAdd(&acc[0], 0ull);
      total.hi = atomicAdd(&acc[1], 0ull);
      if (present || atomicOr(&htouch[h], 0) != 0)
        nins += pull_finish(D, w, d, (present ? cur : 0.0) + fx_to_double(total, L), true,
                            present, c, fmode, qbits);
      acc[0] = 0;
      acc[1] = 0;
      hcnt[h] = 0;
      htouch[h] = 0;
    }
  }
  return nins;
}

template <int BATCH, int GL, typename SH>
__global__ void __launch_bounds__(kBlock)
    pull_heavy_fx_kernel(const int64_t* __restrict__ off, const int32_t* __restrict__ col,
                         const PullItem* __restrict__ items, int64_t nitems,
                         const SH* __restrict__ shx, const int32_t* __restrict__ range, int g,
                         Table D, LiteThr c, int fmode, uint32_t* __restrict__ qbits,
                         Fx* __restrict__ hacc, int32_t* __restrict__ hcnt,
                         int32_t* __restrict__ htouch, Counters* C) {
  const int L = round_scale(range, g);
  const uint32_t be0 = (uint32_t)(2047 - range[0]);
  int64_t nins = 0;
  pull_windows<SH>(range, L, [&](auto w) {
    constexpr int W = decltype(w)::value;
    // shares over any range are rare: a short batch keeps the registers of the
    // others
    constexpr int B = W == 0 && sizeof(SH) == 8 ? 4 : BATCH;
    nins = pull_heavy_fx_body<W, B, GL, SH>(off, col, items, nitems, shx, be0, L, D, c, fmode,
                                            qbits, hacc, hcnt, htouch);
  });
  flush_count(nins, &C->inserted);
}

template <typename SH>
__global__ void pull_light_fx_kernel(LightView V, const SH* __restrict__ shx,
                                     const int32_t* __restrict__ range, int g, Table D, LiteThr c,
                                     int fmode, uint32_t* __restrict__ qbits, Counters* C) {
  const int L = round_scale(range, g);
  const uint32_t be0 = (uint32_t)(2047 - range[0]);
  int64_t nins = 0;
  pull_windows<SH>(range, L, [&](auto w) {
    nins = pull_light_fx_body<decltype(w)::value, SH>(V, shx, be0, L, D, c, fmode, qbits);
  });
  flush_count(nins, &C->inserted);
}

// ---------------------------------------------------------------------------
// edgeMap, deterministic mode.
// ---------------------------------------------------------------------------
// Emits record e of source i: with a self record, local index 0 is
// (v, +0.0) (adding +0.0 to a non-negative value changes nothing) and local
// index q >= 1 is edge q-1; without, local index q is edge q.
__global__ void __launch_bounds__(kBlock)
    emit_records_kernel(const int32_t* __restrict__ col, const int32_t* __restrict__ fv,
                        const double* __restrict__ share, const int64_t* __restrict__ epos,
                        const int64_t* __restrict__ foff, int64_t nf, int64_t R, int self_rec,
                        uint32_t* __restrict__ rkey, double* __restrict__ rval) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  int64_t e0 = warp * 32 * kEdgeItems;  // the tile's first record
  warp_edges<kEdgeItems>(epos, foff, nf, R, warp, nwarps, [&](const int32_t* src,
                                                              const int64_t* at) {
#pragma unroll
    for (int k = 0; k < kEdgeItems; k++) {
      if (src[k] < 0) continue;
      const int64_t e = e0 + 32 * k + lane;
      if (self_rec && at[k] == foff[src[k]]) {
        rkey[e] = (uint32_t)fv[src[k]];
        rval[e] = 0.0;
      } else {
        rkey[e] = (uint32_t)col[at[k] - (self_rec ? 1 : 0)];
        rval[e] = share[src[k]];
      }
    }
    e0 += nwarps * 32 * kEdgeItems;
  });
}

__global__ void head_flags_kernel(const uint32_t* __restrict__ rkey, int64_t R,
                                  int64_t* __restrict__ flag) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < R;
       e += (int64_t)gridDim.x * blockDim.x)
    flag[e] = (e == 0 || rkey[e] != rkey[e - 1]) ? 1 : 0;
}

// flag[] was scanned (exclusive) into segid[]; heads record their start.
__global__ void head_starts_kernel(const uint32_t* __restrict__ rkey, int64_t R,
                                   const int64_t* __restrict__ segid,
                                   int64_t* __restrict__ segstart) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < R;
       e += (int64_t)gridDim.x * blockDim.x)
    if (e == 0 || rkey[e] != rkey[e - 1]) segstart[segid[e]] = e;
}

// One thread per destination run: left fold from the current table value,
// in ascending source order (the order of the run after the stable sort).
// Runs longer than kFoldLong records (a hub destination) are not folded by
// one thread: fold_kernel resolves their slot and lists them, and
// fold_long_kernel folds each with a warp, 256 records at a time, with the
// binade scan of fold_batch (same bits as the sequential fold).
constexpr int64_t kFoldLong = 64;

__global__ void fold_kernel(const uint32_t* __restrict__ rkey, const double* __restrict__ rval,
                            int64_t R, const int64_t* __restrict__ segstart, int64_t nseg,
                            Table D, const int32_t* __restrict__ deg, double c, int fmode,
                            int64_t* __restrict__ qflag, int32_t* __restrict__ segv,
                            int32_t* __restrict__ segslot, int64_t* __restrict__ longs,
                            int32_t* __restrict__ nlong, Counters* C) {
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nseg;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t sg = base + threadIdx.x;
    int ins = 0;
    bool is_long = false;
    if (sg < nseg) {
      const int64_t b = segstart[sg];
      const int64_t e = sg + 1 < nseg ? segstart[sg + 1] : R;
      const int32_t w = (int32_t)rkey[b];
      const int64_t slot = tb_find_or_insert(D, w, &ins, &C->err);
      int64_t q = 0;
      if (slot >= 0 && e - b > kFoldLong) {
        is_long = true;  // folded by fold_long_kernel, which also sets qflag
      } else if (slot >= 0) {
        double acc = *tb_val(D, slot);
        for (int64_t k = b; k < e; k++) acc = acc + rval[k];
        *tb_val(D, slot) = acc;
        if (fmode == kFmThreshold) q = acc >= c * (double)deg[w] ? 1 : 0;
        else if (fmode == kFmInserted) q = 1;
      }
      if (!is_long) qflag[sg] = q;
      segv[sg] = w;
      segslot[sg] = (int32_t)slot;
    }
    // warp-aggregated append of the long runs
    const unsigned active = __activemask();
    const unsigned m = __ballot_sync(active, is_long);
    if (m) {
      const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
      int at = 0;
      if (lane == leader) at = atomicAdd(nlong, __popc(m));
      at = __shfl_sync(active, at, leader);
      if (is_long) longs[at + __popc(m & ((1u << lane) - 1))] = sg;
    }
    count_inserted(ins, &C->inserted);
  }
}

__global__ void __launch_bounds__(kBlock)
    fold_long_kernel(const double* __restrict__ rval, int64_t R,
                     const int64_t* __restrict__ segstart, int64_t nseg,
                     const int64_t* __restrict__ longs, const int32_t* __restrict__ nlong,
                     Table D, const int32_t* __restrict__ deg, double c, int fmode,
                     int64_t* __restrict__ qflag, const int32_t* __restrict__ segv,
                     const int32_t* __restrict__ segslot) {
  const int lane = threadIdx.x & 31;
  const int64_t warp0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t nl = *nlong;
  for (int64_t i = warp0; i < nl; i += nwarps) {
    const int64_t sg = longs[i];
    const int64_t b = segstart[sg];
    const int64_t e = sg + 1 < nseg ? segstart[sg + 1] : R;
    const int32_t w = segv[sg];
    const int64_t slot = segslot[sg];
    double acc = *tb_val(D, slot);  // the same in every lane
    for (int64_t k0 = b; k0 < e; k0 += 256) {
      double v[8];
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const int64_t k = k0 + 8 * lane + j;
        v[j] = k < e ? rval[k] : 0.0;  // +0.0 past the run adds nothing
      }
      acc = fold_batch(acc, v, lane);
    }
    if (lane == 0) {
      *tb_val(D, slot) = acc;
      int64_t q = 0;
      if (fmode == kFmThreshold) q = acc >= c * (double)deg[w] ? 1 : 0;
      else if (fmode == kFmInserted) q = 1;
      qflag[sg] = q;
    }
  }
}

// Order-preserving compaction of the qualifying runs into the next frontier.
__global__ void compact_frontier_kernel(const int64_t* __restrict__ qflag,
                                        const int64_t* __restrict__ qpos, int64_t nseg,
                                        const int32_t* __restrict__ segv,
                                        const int32_t* __restrict__ segslot,
                                        const int32_t* __restrict__ deg, int32_t* nfv,
                                        int32_t* nfs, int32_t ncap, Counters* C) {
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nseg;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t sg = base + threadIdx.x;
    int64_t d = 0;
    if (sg < nseg && qflag[sg]) {
      const int64_t pos = qpos[sg];
      if (pos < ncap) {
        nfv[pos] = segv[sg];
        nfs[pos] = segslot[sg];
      } else {
        atomicOr(&C->err, kErrFrontierOverflow);
      }
      d = deg[segv[sg]];
    }
    // integer sum of degrees: order-independent
    const unsigned active = __activemask();
    unsigned long long lo = __reduce_add_sync(active, (unsigned)(d & 0xFFFF));
    unsigned long long hi = __reduce_add_sync(active, (unsigned)(d >> 16));
    if ((threadIdx.x & 31) == __ffs(active) - 1 && (lo | hi))
      atomicAdd((unsigned long long*)&C->next_edges, lo + (hi << 16));
  }
}

__global__ void set_counter_size_kernel(Counters* C, const int64_t* total) {
  C->next_size = (int32_t)*total;
}

__global__ void init_seed_kernel(Table T, int32_t x, double r0, int32_t* fv, int32_t* fs,
                                 Counters* C) {
  int ins = 0;
  int64_t s = tb_find_or_insert(T, x, &ins, &C->err);
  if (s >= 0) *tb_val(T, s) = r0;
  fv[0] = x;
  fs[0] = (int32_t)s;
}

// Seed set: seeds (ascending, distinct) with their initial residuals.
__global__ void init_seeds_kernel(Table T, const int32_t* __restrict__ x,
                                  const double* __restrict__ r0, int64_t k, int32_t* fv,
                                  int32_t* fs, Counters* C) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k;
       i += (int64_t)gridDim.x * blockDim.x) {
    int ins = 0;
    const int64_t s = tb_find_or_insert(T, x[i], &ins, &C->err);
    if (s >= 0) *tb_val(T, s) = r0[i];
    fv[i] = x[i];
    fs[i] = (int32_t)s;
  }
}

// beta-fraction rounds: order the frontier by r/d descending, ties by
// ascending id (sort by id, then stably by the key 0x7FF...F - bits(r/d)).
__global__ void sel_ids_kernel(const int32_t* __restrict__ fv, int64_t nf,
                               uint32_t* __restrict__ key, int32_t* __restrict__ pos) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf;
       i += (int64_t)gridDim.x * blockDim.x) {
    key[i] = (uint32_t)fv[i];
    pos[i] = (int32_t)i;
  }
}

__global__ void sel_keys_kernel(const int32_t* __restrict__ fv, const int32_t* __restrict__ fs,
                                const int32_t* __restrict__ pos, int64_t nf, Table T,
                                const int32_t* __restrict__ deg, uint64_t* __restrict__ key) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t j = pos[i];
    const double r = fs[j] >= 0 ? *tb_val(T, fs[j]) : 0.0;
    const double kv = r / (double)deg[fv[j]];
    key[i] = 0x7FFFFFFFFFFFFFFFull - ((uint64_t)__double_as_longlong(kv) & 0x7FFFFFFFFFFFFFFFull);
  }
}

// The first m in the order push (written with their ids as keys, to be
// sorted ascending), the rest stay (rv/rs).
__global__ void sel_split_kernel(const int32_t* __restrict__ fv, const int32_t* __restrict__ fs,
                                 const int32_t* __restrict__ pos, int64_t nf, int64_t m,
                                 uint32_t* __restrict__ sv, int32_t* __restrict__ ss,
                                 int32_t* __restrict__ rv, int32_t* __restrict__ rs) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t j = pos[i];
    if (i < m) {
      sv[i] = (uint32_t)fv[j];
      ss[i] = fs[j];
    } else {
      rv[i - m] = fv[j];
      rs[i - m] = fs[j];
    }
  }
}

__global__ void copy_frontier_kernel(const uint32_t* __restrict__ sv,
                                     const int32_t* __restrict__ ss, int64_t m,
                                     const int32_t* __restrict__ deg, int32_t* fv, int32_t* fs,
                                     unsigned long long* edges) {
  unsigned long long e = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    fv[i] = (int32_t)sv[i];
    fs[i] = ss[i];
    e += (unsigned long long)deg[sv[i]];
  }
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0 && e) atomicAdd(edges, e);
}

// Next frontier = the round's qualifying vertices together with the
// candidates that did not push and still have r >= eps d (a seed is on the
// first frontier whatever its residual; afterwards only the threshold
// counts): concatenated, sorted by id, duplicates dropped (a waiting
// candidate that was pushed to may be in both).  A dropped one gets the key
// 0xFFFFFFFF (no vertex id), which sorts last.
__global__ void cat_frontier_kernel(const int32_t* __restrict__ av, const int32_t* __restrict__ as,
                                    int64_t na, const int32_t* __restrict__ bv,
                                    const int32_t* __restrict__ bs, int64_t nb, Table T,
                                    const int32_t* __restrict__ deg, double eps,
                                    uint32_t* __restrict__ kv, int32_t* __restrict__ ks) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < na + nb;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i < na) {
      kv[i] = (uint32_t)av[i];
      ks[i] = as[i];
    } else {
      const int32_t v = bv[i - na], s = bs[i - na];
      const bool keep = s >= 0 && *tb_val(T, s) >= eps * (double)deg[v];
      kv[i] = keep ? (uint32_t)v : 0xFFFFFFFFu;
      ks[i] = s;
    }
  }
}

__global__ void uniq_flags_kernel(const uint32_t* __restrict__ kv, int64_t n,
                                  int64_t* __restrict__ flag) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    flag[i] = (kv[i] != 0xFFFFFFFFu && (i == 0 || kv[i] != kv[i - 1])) ? 1 : 0;
}

__global__ void uniq_write_kernel(const uint32_t* __restrict__ kv, const int32_t* __restrict__ ks,
                                  const int64_t* __restrict__ flag, const int64_t* __restrict__ pos,
                                  int64_t n, const int32_t* __restrict__ deg, int32_t* fv,
                                  int32_t* fs, unsigned long long* edges) {
  unsigned long long e = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (!flag[i]) continue;
    fv[pos[i]] = (int32_t)kv[i];
    fs[pos[i]] = ks[i];
    e += (unsigned long long)deg[kv[i]];
  }
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if ((threadIdx.x & 31) == 0 && e) atomicAdd(edges, e);
}

}  // namespace

template <typename SH>
using HeavyKernel = void (*)(const int64_t*, const int32_t*, const PullItem*, int64_t, const SH*,
                             const int32_t*, int, Table, LiteThr, int, uint32_t*, Fx*, int32_t*,
                             int32_t*, Counters*);

// The heavy-vertex gather compiled for a (batch depth, lanes per item) shape.
template <typename SH>
HeavyKernel<SH> heavy_kernel(int batch, int group) {
  if (group == 8)
    return batch == 16 ? pull_heavy_fx_kernel<16, 8, SH> : pull_heavy_fx_kernel<8, 8, SH>;
  if (group == 16)
    return batch == 16 ? pull_heavy_fx_kernel<16, 16, SH> : pull_heavy_fx_kernel<8, 16, SH>;
  return batch == 16 ? pull_heavy_fx_kernel<16, 32, SH>
         : batch == 4 ? pull_heavy_fx_kernel<4, 32, SH>
                      : pull_heavy_fx_kernel<kPullBatch, 32, SH>;
}

// ---------------------------------------------------------------------------
// Host driver
// ---------------------------------------------------------------------------
namespace {

int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }

int light_grid(const lgc_ctx* ctx, const LightView& V) {
  return (int)min64(ceil_div(V.threads(), kBlock), ctx->sms * 32);
}

// Sets of a graph of up to kDenseSmall vertices are dense from the start
// (automatic form): clearing 16 bytes a vertex costs 4 us at that size,
// growing and converting a table on the way 40 us and more.  For contexts that
// run device rounds: the request loop's workers, many at once, take memory as
// their requests were admitted by (request_bytes), from small tables up.
constexpr int64_t kDenseSmall = int64_t{1} << 20;
// Keys a table has room for ahead of the device-driven rounds.
constexpr int64_t kRoomKeys = 16384;

// Slots of a hashed table for device-driven rounds that has to take `need`
// keys: room for `times` as many, so that the rounds to come fit as well, up
// to `limit` slots, beyond that for twice as many.  Room is cleared (24 bytes
// a slot, as much again in per-slot sums, three fresh sets a launch) and read
// through at the end; too little costs a launch and a rehash, 50 us.  Calls on
// R-MAT graphs, us, without limits and with these: Nibble 2^22 vertices, eps
// 1e-7 581 and 513, 2^24, 1e-6 504 and 383, 2^26, 1e-7 669 and 750; PR-Nibble
// 2^22, 3e-7 315 and 317 (2^20 slots: 353), 2^24, 1e-7 405 and 427, 2^26, 1e-7
// 720 and 524; HK-PR 2^24, 1e-6 615 and 569, 2^26, 1e-7 2535 and 2237.
constexpr int64_t kRoomKept = int64_t{1} << 22;
constexpr int64_t kRoomFresh = int64_t{1} << 20;
int64_t room_slots(int64_t need, int64_t n, int64_t times, int64_t limit) {
  constexpr int64_t kMostSlots = int64_t{1} << 31;  // of any table
  const int64_t least = pow2_at_least(2 * min64(n, need));
  const int64_t ahead = pow2_at_least(2 * min64(n, std::max<int64_t>(times * need, kRoomKeys)));
  const int64_t twice = pow2_at_least(2 * min64(n, 2 * need));
  return std::max(least, min64(kMostSlots, min64(ahead, std::max(limit, twice))));
}

bool dense_small(const lgc_ctx* ctx, int64_t n) {
  return ctx->device_rounds && ctx->table_form == 0 && n >= 1024 && n <= kDenseSmall;
}

struct Frontier {
  DBuf<int32_t> v, s;
  int64_t size = 0, edges = 0;
  void release(lgc_ctx* ctx) {
    v.release(ctx);
    s.release(ctx);
  }
};

struct PushWork {
  lgc_ctx* ctx;
  lgc_graph* g;
  Frontier F, G;
  DBuf<double> share;
  DBuf<int64_t> cnt, epos, foff;
  DBuf<uint32_t> rk, rk2;
  DBuf<double> rv, rv2;
  DBuf<int64_t> flag, segid, segstart, qflag, qpos;
  DBuf<int32_t> segv, segslot;
  DBuf<int64_t> longs;  // runs folded by a warp
  DBuf<int32_t> nlong;
  DBuf<int64_t> total;  // one device int64
  // pull rounds: per-vertex frontier share (membership encoded), qualify bitmap
  DBuf<double> psh;
  DBuf<uint32_t> pq;
  DBuf<Fx> pshx;                   // atomic mode: per-vertex fixed-point shares
  DBuf<int32_t> prange;            // atomic mode: exponent range of the shares
  DBuf<Fx> phacc;                  // per heavy vertex: partial sums of its items
  DBuf<int32_t> phcnt, phtouch;    // per heavy vertex: items done, any frontier neighbour
  // deterministic pull of big vertices: per segment sum, member flag,
  // predicted binade, composed step
  DBuf<double> dsum, dkept;
  DBuf<int32_t> dany, dpred;
  DBuf<FoldStep> dstep;
  bool pull_ready = false;
  // beta-fraction rounds: the candidates that did not push, sort scratch
  Frontier U;
  DBuf<uint64_t> selk, selk2;
  DBuf<uint32_t> selv, selv2;
  DBuf<int32_t> seli, seli2;
  DBuf<unsigned long long> selcnt;
  // device-driven rounds
  RoundsMem rmem;
  // graphs with sinks: the push's arrays in another order
  DBuf<double> share2;
  DBuf<int64_t> epos2, foff2, has;
  DBuf<Recip> recip;  // HK-PR pull rounds: 1 / ((j + 1) d) by degree
  lgc_stats st{};
  explicit PushWork(lgc_ctx* c, lgc_graph* gr) : ctx(c), g(gr) {}
  ~PushWork() {
    F.release(ctx);
    G.release(ctx);
    U.release(ctx);
    selk.release(ctx);
    selk2.release(ctx);
    selv.release(ctx);
    selv2.release(ctx);
    seli.release(ctx);
    seli2.release(ctx);
    selcnt.release(ctx);
    dsum.release(ctx);
    dkept.release(ctx);
    dany.release(ctx);
    dpred.release(ctx);
    dstep.release(ctx);
    rmem.release(ctx);
    share2.release(ctx);
    epos2.release(ctx);
    foff2.release(ctx);
    has.release(ctx);
    recip.release(ctx);
    share.release(ctx);
    cnt.release(ctx);
    epos.release(ctx);
    foff.release(ctx);
    rk.release(ctx);
    rk2.release(ctx);
    rv.release(ctx);
    rv2.release(ctx);
    flag.release(ctx);
    segid.release(ctx);
    segstart.release(ctx);
    qflag.release(ctx);
    qpos.release(ctx);
    segv.release(ctx);
    segslot.release(ctx);
    longs.release(ctx);
    nlong.release(ctx);
    total.release(ctx);
    psh.release(ctx);
    pshx.release(ctx);
    prange.release(ctx);
    pq.release(ctx);
    phacc.release(ctx);
    phcnt.release(ctx);
    phtouch.release(ctx);
  }

  int reset_counters() {
    LGC_CUDA_TRY(cudaMemsetAsync(ctx->d_counters, 0, sizeof(Counters), ctx->stream));
    return LGC_OK;
  }
  int read_counters(Counters* out) {
    LGC_CUDA_TRY(cudaMemcpyAsync(ctx->h_counters, ctx->d_counters, sizeof(Counters),
                                 cudaMemcpyDeviceToHost, ctx->stream));
    LGC_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
    LGC_TRY(sort_check(ctx));
    *out = *ctx->h_counters;
    if (out->err & kErrTableFull) return LGC_ETABLEFULL;
    if (out->err & kErrFrontierOverflow) return LGC_ETABLEFULL;
    return LGC_OK;
  }
  int reserve_frontier_scratch(int64_t nf) {
    LGC_TRY(share.reserve(ctx, nf));
    LGC_TRY(cnt.reserve(ctx, nf));
    LGC_TRY(epos.reserve(ctx, nf));
    LGC_TRY(foff.reserve(ctx, nf));
    LGC_TRY(total.reserve(ctx, 1));
    return LGC_OK;
  }
  int reserve_next(int64_t cap) {
    LGC_TRY(G.v.reserve(ctx, cap));
    LGC_TRY(G.s.reserve(ctx, cap));
    return LGC_OK;
  }
  void record_trace() {
    if (!ctx->trace) return;
    size_t at = ctx->trace_ids.size();
    ctx->trace_ids.resize(at + F.size);
    if (F.size)
      cudaMemcpyAsync(ctx->trace_ids.data() + at, F.v.ptr, 4 * F.size, cudaMemcpyDeviceToHost,
                      ctx->stream);
    cudaStreamSynchronize(ctx->stream);
    ctx->trace_sizes.push_back(F.size);
  }

  // The push's sources without edges behind the others.
  int sinks_last() {
    cudaStream_t s = ctx->stream;
    const int64_t nf = F.size;
    LGC_TRY(share2.reserve(ctx, nf));
    LGC_TRY(epos2.reserve(ctx, nf));
    LGC_TRY(foff2.reserve(ctx, nf));
    LGC_TRY(has.reserve(ctx, nf + 1));
    has_edges_kernel<<<grid_for(nf), kBlock, 0, s>>>(cnt.ptr, nf, has.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_TRY(scan_i64(ctx, has.ptr, has.ptr, nf, false, has.ptr + nf));
    sinks_last_kernel<<<grid_for(nf), kBlock, 0, s>>>(nf, cnt.ptr, has.ptr, has.ptr + nf,
                                                      total.ptr, share.ptr, epos.ptr, foff.ptr,
                                                      share2.ptr, epos2.ptr, foff2.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_CUDA_TRY(cudaGetLastError());
    std::swap(share, share2);
    std::swap(epos, epos2);
    std::swap(foff, foff2);
    return LGC_OK;
  }

  // edgeMap + filter into table D.  Records per source are cnt[] (scanned
  // into epos by the caller's vertexMap step).  Returns the counters.
  int edge_phase(const Table& D, double c, int fmode, bool det, bool self_rec, int64_t nrec,
                 Counters* out, bool bulk = false) {
    cudaStream_t s = ctx->stream;
    const int64_t nf = F.size;
    const int32_t ncap = (int32_t)G.v.cap;
    // algorithmic bytes: 24 per pushed edge (col 4, key 4, value read-modify-write 16),
    // 24 per frontier source staged (epos, off, share), 8 per next-frontier entry
    const double alg_bytes = 24.0 * (double)(nrec - (self_rec && det ? nf : 0)) + 24.0 * nf;
    // (with a record of its own every source has one)
    if (g->sinks && nrec > 0 && !(self_rec && det)) LGC_TRY(sinks_last());
    if (bulk) {
      if (nrec > 0) {
        int64_t tiles = ceil_div(nrec, kEdgeTile);
        int grid = (int)(tiles < (ctx->sms * 16) ? tiles : (ctx->sms * 16));
        {
          ProfScope ps(ctx, LGC_PROF_EDGEMAP, alg_bytes);
          emap_red_kernel<<<grid, kBlock, 0, s>>>(g->col, share.ptr, epos.ptr, foff.ptr, nf, nrec,
                                                   total.ptr, g->hot, D, fmode == kFmNone ? 1 : 0,
                                                   ctx->d_counters);
          LGC_COUNT_LAUNCH(ctx);
        }
        LGC_CUDA_TRY(cudaGetLastError());
      }
      if (fmode != kFmNone) {  // the qualifying keys in ascending id, with their degrees
        const int64_t words = (g->n + 31) / 32;
        LGC_TRY(words_compact(ctx, DenseQualWord{D, g->deg, g->n, lite_thr(c), fmode,
                                                 &ctx->d_counters->inserted}, nullptr, words,
                              FrontierOut{g->deg, G.v.ptr, G.s.ptr, ncap, ctx->d_counters}));
      }
      int st = read_counters(out);
      if (ctx->profile && nrec > 0 && !ctx->prof_pending.empty())
        ctx->prof_pending.back().bytes += 8.0 * out->next_size;
      return st;
    }
    if (!det) {
      if (nrec > 0) {
        int64_t tiles = ceil_div(nrec, kEdgeTile);
        int grid = (int)(tiles < (ctx->sms * 16) ? tiles : (ctx->sms * 16));
        ProfScope ps(ctx, LGC_PROF_EDGEMAP, alg_bytes);
        emap_atomic_kernel<<<grid, kBlock, 0, s>>>(g->col, g->deg, share.ptr, epos.ptr, foff.ptr,
                                                    nf, nrec, total.ptr, g->hot, D, c, fmode, G.v.ptr,
                                                    G.s.ptr, ncap, ctx->d_counters);
        LGC_COUNT_LAUNCH(ctx);
        LGC_CUDA_TRY(cudaGetLastError());
      }
      int st = read_counters(out);
      if (ctx->profile && nrec > 0 && !ctx->prof_pending.empty())
        ctx->prof_pending.back().bytes += 8.0 * out->next_size;
      return st;
    }
    // deterministic: emit, stable sort by destination, fold, compact
    LGC_TRY(rk.reserve(ctx, nrec));
    LGC_TRY(rk2.reserve(ctx, nrec));
    LGC_TRY(rv.reserve(ctx, nrec));
    LGC_TRY(rv2.reserve(ctx, nrec));
    LGC_TRY(flag.reserve(ctx, nrec));
    LGC_TRY(segid.reserve(ctx, nrec));
    if (nrec > 0) {
      int64_t tiles = ceil_div(nrec, kEdgeTile);
      int grid = (int)(tiles < (ctx->sms * 16) ? tiles : (ctx->sms * 16));
      ProfScope ps(ctx, LGC_PROF_DET_EDGE, alg_bytes);
      emit_records_kernel<<<grid, kBlock, 0, s>>>(g->col, F.v.ptr, share.ptr, epos.ptr, foff.ptr,
                                                   nf, nrec, self_rec ? 1 : 0, rk.ptr, rv.ptr);
      LGC_COUNT_LAUNCH(ctx);
      LGC_CUDA_TRY(cudaGetLastError());
      LGC_TRY(radix_sort_u32_f64(ctx, rk.ptr, rv.ptr, rk2.ptr, rv2.ptr, nrec, bits_for(g->n)));
      head_flags_kernel<<<grid_for(nrec), kBlock, 0, s>>>(rk.ptr, nrec, flag.ptr);
      LGC_COUNT_LAUNCH(ctx);
      LGC_TRY(scan_i64(ctx, flag.ptr, segid.ptr, nrec, false, total.ptr));
    }
    int64_t nseg = 0;
    if (nrec > 0) {
      LGC_CUDA_TRY(cudaMemcpyAsync(&ctx->h_counters->aux, total.ptr, 8, cudaMemcpyDeviceToHost, s));
      LGC_CUDA_TRY(cudaStreamSynchronize(s));
      nseg = ctx->h_counters->aux;
    }
    LGC_TRY(segstart.reserve(ctx, nseg));
    LGC_TRY(qflag.reserve(ctx, nseg));
    LGC_TRY(qpos.reserve(ctx, nseg));
    LGC_TRY(segv.reserve(ctx, nseg));
    LGC_TRY(segslot.reserve(ctx, nseg));
    if (nseg > 0) {
      ProfScope ps(ctx, LGC_PROF_DET_EDGE, 0.0);
      head_starts_kernel<<<grid_for(nrec), kBlock, 0, s>>>(rk.ptr, nrec, segid.ptr, segstart.ptr);
      LGC_COUNT_LAUNCH(ctx);
      LGC_TRY(longs.reserve(ctx, nseg));
      LGC_TRY(nlong.reserve(ctx, 1));
      LGC_CUDA_TRY(cudaMemsetAsync(nlong.ptr, 0, 4, s));
      fold_kernel<<<grid_for(nseg), kBlock, 0, s>>>(rk.ptr, rv.ptr, nrec, segstart.ptr, nseg, D,
                                                     g->deg, c, fmode, qflag.ptr, segv.ptr,
                                                     segslot.ptr, longs.ptr, nlong.ptr,
                                                     ctx->d_counters);
      LGC_COUNT_LAUNCH(ctx);
      fold_long_kernel<<<ctx->sms * 4, kBlock, 0, s>>>(rv.ptr, nrec, segstart.ptr, nseg,
                                                        longs.ptr, nlong.ptr, D, g->deg, c, fmode,
                                                        qflag.ptr, segv.ptr, segslot.ptr);
      LGC_COUNT_LAUNCH(ctx);
      LGC_CUDA_TRY(cudaGetLastError());
      if (fmode != kFmNone) {
        LGC_TRY(scan_i64(ctx, qflag.ptr, qpos.ptr, nseg, false, total.ptr));
        compact_frontier_kernel<<<grid_for(nseg), kBlock, 0, s>>>(
            qflag.ptr, qpos.ptr, nseg, segv.ptr, segslot.ptr, g->deg, G.v.ptr, G.s.ptr, ncap,
            ctx->d_counters);
        LGC_COUNT_LAUNCH(ctx);
        set_counter_size_kernel<<<1, 1, 0, s>>>(ctx->d_counters, total.ptr);
        LGC_COUNT_LAUNCH(ctx);
        LGC_CUDA_TRY(cudaGetLastError());
      }
    }
    return read_counters(out);
  }

  // The bytes per gathered share of a pull round: atomic mode gathers 16-byte
  // fixed-point records or 8-byte doubles (the graph's tuned choice);
  // deterministic mode always doubles.
  int pull_share_bytes(bool det) const {
    return det ? 8 : (ctx->pull_share ? ctx->pull_share : g->pull_share);
  }

  // The pull rounds' per-vertex arrays (zeroed at first use; every round
  // leaves them zeroed again).
  int pull_reserve(bool det) {
    cudaStream_t s = ctx->stream;
    const int64_t n = g->n, words = (n + 31) / 32;
    if (!pull_ready) {
      LGC_TRY(pq.reserve(ctx, words + 1));
      pull_ready = true;
    }
    const int sb = pull_share_bytes(det);
    if (sb == 8 && !psh.ptr) {
      LGC_TRY(psh.reserve(ctx, n));
      LGC_CUDA_TRY(cudaMemsetAsync(psh.ptr, 0, 8 * n, s));
    }
    if (!det && sb == 16 && !pshx.ptr) {
      LGC_TRY(pshx.reserve(ctx, n));
      LGC_CUDA_TRY(cudaMemsetAsync(pshx.ptr, 0, sizeof(Fx) * n, s));
    }
    if (!det && !prange.ptr) {
      LGC_TRY(prange.reserve(ctx, 2));
      LGC_TRY(phacc.reserve(ctx, g->nheavy + 1));
      LGC_TRY(phcnt.reserve(ctx, g->nheavy + 1));
      LGC_TRY(phtouch.reserve(ctx, g->nheavy + 1));
      LGC_CUDA_TRY(cudaMemsetAsync(phacc.ptr, 0, sizeof(Fx) * (g->nheavy + 1), s));
      LGC_CUDA_TRY(cudaMemsetAsync(phcnt.ptr, 0, 4 * (g->nheavy + 1), s));
      LGC_CUDA_TRY(cudaMemsetAsync(phtouch.ptr, 0, 4 * (g->nheavy + 1), s));
    }
    return LGC_OK;
  }

  // Pull round into the dense table D.  The frontier's shares (share[], from
  // the vertexMap) are scattered into the per-vertex array -- unless the
  // vertexMap wrote them there itself (scattered: 8-byte shares, with the
  // range in atomic mode) --, every vertex gathers (in adjacency order in
  // deterministic mode, heavy vertices by a tree reduction in atomic mode),
  // the qualifying vertices are compacted in ascending id, and the
  // per-vertex array is cleared again (O(|F|)).
  int pull_phase(const Table& D, double c, int fmode, Counters* out, bool det,
                 bool scattered = false) {
    cudaStream_t s = ctx->stream;
    const int64_t n = g->n, words = (n + 31) / 32, nf = F.size;
    LGC_TRY(pull_reserve(det));
    const int sb = pull_share_bytes(det);
    const LiteThr ct = lite_thr(c);
    const int32_t ncap = (int32_t)G.v.cap;
    // sums of at most max_deg terms: max_deg < 2^gb
    int gb = 1;
    while (gb < 62 && (int64_t{1} << gb) <= g->max_deg) gb++;
    if (!scattered && det) {
      pull_scatter_kernel<<<grid_for(nf), kBlock, 0, s>>>(nf, F.v.ptr, share.ptr, psh.ptr, 0);
      LGC_COUNT_LAUNCH(ctx);
    } else if (!scattered) {
      LGC_CUDA_TRY(cudaMemsetAsync(prange.ptr, 0, 8, s));
      const int64_t rb = ceil_div(nf, kBlock);
      const int rg = (int)std::max<int64_t>(1, std::min<int64_t>(rb, ctx->sms * 4));
      share_range_kernel<<<rg, kBlock, 0, s>>>(nf, share.ptr, prange.ptr);
      LGC_COUNT_LAUNCH(ctx);
      if (sb == 8) {
        pull_scatter_kernel<<<grid_for(nf), kBlock, 0, s>>>(nf, F.v.ptr, share.ptr, psh.ptr, 0);
      } else {
        pull_scatter_fx_kernel<<<grid_for(nf), kBlock, 0, s>>>(nf, F.v.ptr, share.ptr, pshx.ptr,
                                                                prange.ptr, gb, 0);
      }
      LGC_COUNT_LAUNCH(ctx);
    }
    {
      ProfScope ps(ctx, det ? LGC_PROF_DET_EDGE : LGC_PROF_PULL,
                   24.0 * (double)F.edges + 24.0 * nf);
      if (det) {
        // every gather ORs its qualifying vertices into the cleared bitmap (and
        // the word after it, the middle gather's slice ticket)
        LGC_CUDA_TRY(cudaMemsetAsync(pq.ptr, 0, 4 * (words + 1), s));
        const LightView light = g->view(1, kPullLight), mid = g->view(kPullLight + 1, kDetBig);
        if (light.end > light.beg) {
          pull_light_kernel<<<light_grid(ctx, light), kBlock, 0, s>>>(
              light, psh.ptr, D, ct, fmode, pq.ptr, ctx->d_counters);
          LGC_COUNT_LAUNCH(ctx);
        }
        if (mid.end > mid.beg) {
          const int mg = (int)min64(ceil_div(mid.threads(), 32), ctx->sms);
          pull_mid_det_kernel<<<mg, kBlock, 0, s>>>(mid, psh.ptr, D, ct, fmode, pq.ptr,
                                                    pq.ptr + words, ctx->d_counters);
          LGC_COUNT_LAUNCH(ctx);
        }
        if (g->nbig > 0) {  // lists longer than kDetBig, folded segment-parallel
          LGC_TRY(dsum.reserve(ctx, g->nsegs));
          LGC_TRY(dany.reserve(ctx, g->nsegs));
          LGC_TRY(dpred.reserve(ctx, g->nsegs));
          LGC_TRY(dstep.reserve(ctx, g->nsegs));
          const int sg = (int)std::min<int64_t>(ceil_div(g->nsegs, kBlock / 32), (ctx->sms * 16));
          const bool keep = g->nsegs <= kDetKeep &&
                            dkept.reserve(ctx, kDetSeg * g->nsegs) == LGC_OK;
          det_seg_sum_kernel<<<sg, kBlock, 0, s>>>(g->col, g->segs, g->nsegs, psh.ptr, dsum.ptr,
                                                   dany.ptr, keep ? dkept.ptr : nullptr);
          LGC_COUNT_LAUNCH(ctx);
          const int vg = (int)std::min<int64_t>(ceil_div(g->nbig, kBlock / 32), (ctx->sms * 16));
          det_seg_predict_kernel<<<vg, kBlock, 0, s>>>(g->big_w, g->big_seg0, g->nbig, D, dsum.ptr,
                                                       dpred.ptr);
          LGC_COUNT_LAUNCH(ctx);
          det_seg_step_kernel<<<sg, kBlock, 0, s>>>(g->col, g->segs, g->nsegs, psh.ptr,
                                                    keep ? dkept.ptr : nullptr, dpred.ptr,
                                                    dstep.ptr);
          LGC_COUNT_LAUNCH(ctx);
          det_seg_verify_kernel<<<vg, kBlock, 0, s>>>(
              g->off, g->col, g->segs, g->big_w, g->big_seg0, g->nbig, psh.ptr,
              keep ? dkept.ptr : nullptr, dpred.ptr, dstep.ptr, dany.ptr, D, ct, fmode, pq.ptr,
              ctx->d_counters);
          LGC_COUNT_LAUNCH(ctx);
        }
      } else {
        // light vertices, then the heavy items, both ORing their vertices into
        // the cleared bitmap; the two in one grid measured slower
        auto gather = [&](auto* shv) {
          using SH = std::remove_const_t<std::remove_pointer_t<decltype(shv)>>;
          const LightView light = g->view(1, g->pull_light);
          if (light.end > light.beg) {
            pull_light_fx_kernel<SH><<<light_grid(ctx, light), kBlock, 0, s>>>(
                light, shv, prange.ptr, gb, D, ct, fmode, pq.ptr, ctx->d_counters);
            LGC_COUNT_LAUNCH(ctx);
          }
          if (g->nitems > 0) {
            const int gw = ctx->pull_group ? ctx->pull_group : g->pull_group;
            const int64_t hb = ceil_div(g->nitems, (kBlock / 32) * (32 / gw));
            const int hg = (int)(hb < (ctx->sms * 16) ? hb : (ctx->sms * 16));
            const int batch = ctx->pull_batch ? ctx->pull_batch : g->pull_batch;
            HeavyKernel<SH> heavy = heavy_kernel<SH>(batch, gw);
            heavy<<<hg, kBlock, 0, s>>>(g->off, g->col, g->items, g->nitems, shv, prange.ptr, gb,
                                        D, ct, fmode, pq.ptr, phacc.ptr, phcnt.ptr, phtouch.ptr,
                                        ctx->d_counters);
            LGC_COUNT_LAUNCH(ctx);
          }
        };
        // both gathers OR their qualifying vertices into the cleared bitmap
        LGC_CUDA_TRY(cudaMemsetAsync(pq.ptr, 0, 4 * words, s));
        if (sb == 8) gather(psh.ptr);
        else gather(pshx.ptr);
      }
    }
    if (fmode != kFmNone)  // the qualifying vertices, in ascending id, with their degrees
      LGC_TRY(bits_compact(ctx, pq.ptr, words, g->deg, G.v.ptr, G.s.ptr, ncap, ctx->d_counters));
    if (sb == 8) {
      pull_scatter_kernel<<<grid_for(nf), kBlock, 0, s>>>(nf, F.v.ptr, share.ptr, psh.ptr, 1);
    } else {
      pull_scatter_fx_kernel<<<grid_for(nf), kBlock, 0, s>>>(nf, F.v.ptr, share.ptr, pshx.ptr,
                                                              prange.ptr, gb, 1);
    }
    LGC_COUNT_LAUNCH(ctx);
    LGC_CUDA_TRY(cudaGetLastError());
    return read_counters(out);
  }

  // keys T takes within load 1/2 (no set has more than n)
  int64_t key_limit(const Table& T) const {
    return T.dense || T.cap >= 2 * g->n ? INT64_MAX : T.cap / 2;
  }
  // The edges from which a round is a pull round (use_pull), automatic policy.
  int64_t pull_min() const {
    if (ctx->table_form == 1 || ctx->pull_policy == 1 || g->n < 1024) return INT64_MAX;
    return g->nnz / 16;
  }
  // PR-Nibble's small rounds on the device (rounds.cu) from the state in F, T
  // and count; afterwards those and st describe the state reached.
  int device_rounds_prnibble(Table& T, int64_t* count, double alpha, double cs, double cn,
                             double eps, int rule, bool det, double beta, int64_t rounds_left) {
    cudaStream_t s = ctx->stream;
    RoundsOut o;
    LGC_TRY(rounds_prnibble(ctx, g, rmem, T, F.v.ptr, F.s.ptr, F.size, F.edges, *count, alpha, cs,
                            cn, eps, rule, det, beta, pull_min(), rounds_left, key_limit(T), &o));
    if (o.rounds == 0) return LGC_OK;  // no room for them: the rounds stay on the host
    LGC_TRY(F.v.reserve(ctx, std::max<int64_t>(o.nf, 1024)));
    LGC_TRY(F.s.reserve(ctx, std::max<int64_t>(o.nf, 1024)));
    if (o.nf > 0) {
      LGC_CUDA_TRY(cudaMemcpyAsync(F.v.ptr, o.v, 4 * o.nf, cudaMemcpyDeviceToDevice, s));
      LGC_CUDA_TRY(cudaMemcpyAsync(F.s.ptr, o.s, 4 * o.nf, cudaMemcpyDeviceToDevice, s));
    }
    F.size = o.nf;
    F.edges = o.E;
    *count = o.count;
    st.rounds += o.rounds;
    st.pushes += o.pushes;
    st.pushed_edges += o.pushed;
    return LGC_OK;
  }

  // Small rounds into fresh sets on the device (rounds.cu): Nibble's (c
  // null) from the vector in S, or HK-PR's from level *j with residuals in S
  // and p in P.  *done counts the rounds run (0: no room for them); S is the
  // set reached (Nibble with *over: the vector returned), F and st follow.
  int device_rounds_fresh(Table& S, Table& Sn, Table* P, int64_t* pcount, int64_t* count,
                          const RoundsFresh& q, bool det, int64_t rounds_left, int64_t* done,
                          bool* over) {
    cudaStream_t s = ctx->stream;
    *done = 0;
    *over = false;
    // fresh sets with room for more than this round's keys, in the smaller form
    // (a round that would not fit returns to the host, which comes back with
    // bigger ones); dense ones where they are cheap to clear
    const int64_t n = g->n, need = std::min<int64_t>(n, F.size + F.edges);
    const int64_t cap = room_slots(need, n, 8, kRoomFresh);
    const bool dense = want_dense(ctx, need, n) || dense_small(ctx, n) ||
                       (ctx->table_form == 0 && n >= 1024 && 16 * cap >= 8 * n);
    Table T[4];
    T[3] = S;
    int st_ = LGC_OK;
    for (int k = 0; k < 3 && st_ == LGC_OK; k++)
      st_ = dense ? table_create_dense(ctx, &T[k], n, false) : table_create(ctx, &T[k], cap, false);
    RoundsOut o;
    if (st_ == LGC_OK)
      st_ = rounds_fresh(ctx, g, rmem, q, T, P, pcount ? *pcount : 0, F.v.ptr, F.s.ptr, F.size,
                         F.edges, det, pull_min(), rounds_left, key_limit(T[0]),
                         P ? key_limit(*P) : 0, &o);
    else if (st_ == LGC_ENOMEM) {  // no room for the sets: the rounds stay on the host
      rmem.give_up(ctx);
      st_ = LGC_OK;
    }
    if (st_ != LGC_OK || o.rounds == 0) {
      for (int k = 0; k < 3; k++) table_destroy(ctx, &T[k]);
      return st_;
    }
    *done = o.rounds;
    *over = o.nf == 0;
    for (int k = 0; k < 3; k++)
      if (k != o.tab) table_destroy(ctx, &T[k]);
    if (o.tab != 3) {
      table_destroy(ctx, &S);
      table_destroy(ctx, &Sn);
      S = T[o.tab];
    }
    *count = o.count;
    if (pcount) *pcount = o.pcount;
    st.rounds += o.rounds;
    st.pushes += o.pushes;
    st.pushed_edges += o.pushed;
    LGC_TRY(F.v.reserve(ctx, std::max<int64_t>(o.nf, 1024)));
    LGC_TRY(F.s.reserve(ctx, std::max<int64_t>(o.nf, 1024)));
    if (o.nf > 0) {
      LGC_CUDA_TRY(cudaMemcpyAsync(F.v.ptr, o.v, 4 * o.nf, cudaMemcpyDeviceToDevice, s));
      LGC_CUDA_TRY(cudaMemcpyAsync(F.s.ptr, o.s, 4 * o.nf, cudaMemcpyDeviceToDevice, s));
    }
    F.size = o.nf;
    F.edges = o.E;
    return LGC_OK;
  }

  // beta-fraction rounds: keeps in F the first m candidates by r/d
  // descending (ties by ascending id), in ascending id, and moves the others
  // to U (they stay candidates).
  int select_top(const Table& T, int64_t m) {
    cudaStream_t s = ctx->stream;
    const int64_t nf = F.size, E0 = F.edges;
    const int vb = bits_for(g->n);
    LGC_TRY(selv.reserve(ctx, nf));
    LGC_TRY(selv2.reserve(ctx, nf));
    LGC_TRY(seli.reserve(ctx, nf));
    LGC_TRY(seli2.reserve(ctx, nf));
    LGC_TRY(selk.reserve(ctx, nf));
    LGC_TRY(selk2.reserve(ctx, nf));
    LGC_TRY(selcnt.reserve(ctx, 2));
    LGC_TRY(U.v.reserve(ctx, nf));
    LGC_TRY(U.s.reserve(ctx, nf));
    sel_ids_kernel<<<grid_for(nf), kBlock, 0, s>>>(F.v.ptr, nf, selv.ptr, seli.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_TRY(radix_sort_u32_i32(ctx, selv.ptr, seli.ptr, selv2.ptr, seli2.ptr, nf, vb));
    sel_keys_kernel<<<grid_for(nf), kBlock, 0, s>>>(F.v.ptr, F.s.ptr, seli.ptr, nf, T, g->deg,
                                                     selk.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_TRY(radix_sort_u64_i32(ctx, selk.ptr, seli.ptr, selk2.ptr, seli2.ptr, nf, 64));
    sel_split_kernel<<<grid_for(nf), kBlock, 0, s>>>(F.v.ptr, F.s.ptr, seli.ptr, nf, m, selv.ptr,
                                                      seli2.ptr, U.v.ptr, U.s.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_TRY(radix_sort_u32_i32(ctx, selv.ptr, seli2.ptr, selv2.ptr, seli.ptr, m, vb));
    LGC_CUDA_TRY(cudaMemsetAsync(selcnt.ptr, 0, 8, s));
    copy_frontier_kernel<<<grid_for(m), kBlock, 0, s>>>(selv.ptr, seli2.ptr, m, g->deg, F.v.ptr,
                                                         F.s.ptr, selcnt.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, selcnt.ptr, 8, cudaMemcpyDeviceToHost, s));
    LGC_CUDA_TRY(cudaStreamSynchronize(s));
    F.size = m;
    F.edges = ctx->h_scratch[0];
    U.size = nf - m;
    U.edges = E0 - F.edges;
    return LGC_OK;
  }

  // G (the round's next frontier) united with U: sorted by id, duplicates
  // dropped.
  int merge_rest(const Table& T, double eps) {
    if (U.size == 0) return LGC_OK;
    cudaStream_t s = ctx->stream;
    const int64_t na = G.size, nb = U.size, tot = na + nb;
    LGC_TRY(selv.reserve(ctx, tot));
    LGC_TRY(selv2.reserve(ctx, tot));
    LGC_TRY(seli.reserve(ctx, tot));
    LGC_TRY(seli2.reserve(ctx, tot));
    LGC_TRY(flag.reserve(ctx, tot));
    LGC_TRY(qpos.reserve(ctx, tot));
    LGC_TRY(selcnt.reserve(ctx, 2));
    cat_frontier_kernel<<<grid_for(tot), kBlock, 0, s>>>(G.v.ptr, G.s.ptr, na, U.v.ptr, U.s.ptr,
                                                          nb, T, g->deg, eps, selv.ptr, seli.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_TRY(radix_sort_u32_i32(ctx, selv.ptr, seli.ptr, selv2.ptr, seli2.ptr, tot, 32));
    uniq_flags_kernel<<<grid_for(tot), kBlock, 0, s>>>(selv.ptr, tot, flag.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_TRY(scan_i64(ctx, flag.ptr, qpos.ptr, tot, false, (int64_t*)selcnt.ptr + 1));
    // G's entries are in selv/seli now: its buffers may be replaced
    LGC_TRY(G.v.reserve(ctx, tot));
    LGC_TRY(G.s.reserve(ctx, tot));
    LGC_CUDA_TRY(cudaMemsetAsync(selcnt.ptr, 0, 8, s));
    uniq_write_kernel<<<grid_for(tot), kBlock, 0, s>>>(selv.ptr, seli.ptr, flag.ptr, qpos.ptr, tot,
                                                        g->deg, G.v.ptr, G.s.ptr, selcnt.ptr);
    LGC_COUNT_LAUNCH(ctx);
    LGC_CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, selcnt.ptr, 16, cudaMemcpyDeviceToHost, s));
    LGC_CUDA_TRY(cudaStreamSynchronize(s));
    G.edges = ctx->h_scratch[0];
    G.size = ctx->h_scratch[1];
    U.size = 0;
    U.edges = 0;
    return LGC_OK;
  }


  void swap_frontiers() {
    std::swap(F.v, G.v);
    std::swap(F.s, G.s);
    F.size = G.size;
    F.edges = G.edges;
    G.size = 0;
    G.edges = 0;
  }
};

int vgrid(const lgc_ctx* ctx, int64_t nf) {
  int64_t g = ceil_div(nf, kBlock);
  if (g > (ctx->sms * 32)) g = (ctx->sms * 32);
  return (int)(g < 1 ? 1 : g);
}


// Bulk rounds (atomic mode): the destination is dense and the round pushes at
// least n/32 edges, so a filter pass over the n-bit presence bitmap costs no
// more than a constant times the round's own work.
bool use_bulk(bool det, const Table& D, int64_t round_edges, int64_t n) {
  return !det && D.dense && round_edges >= n / 32;
}

// Pull rounds: when the frontier's edges are at least 1/16 of the graph's,
// gathering over every vertex costs no more than a constant times the push
// it replaces, and it needs neither atomics nor (deterministic mode) records
// and a sort.  The destination must be (made) dense.
bool use_pull(const lgc_ctx* ctx, const lgc_graph* g, int64_t round_edges) {
  if (ctx->table_form == 1 || ctx->pull_policy == 1) return false;
  if (ctx->pull_policy == 2) return true;
  return g->n >= 1024 && round_edges >= g->nnz / 16;
}

// An empty dense table over n vertices (reusing the allocation if it is one).
int fresh_dense(lgc_ctx* ctx, Table* T, int64_t n) {
  if (T->dense && T->cap == n && !T->p) return table_clear(ctx, T);
  table_destroy(ctx, T);
  return table_create_dense(ctx, T, n, false);
}

// An empty dense table for a pull round's destination: only the presence
// bitmap is cleared, since the gathers set a vertex's value when they make it
// a key and never read the value of a non-key, and the table's later readers
// read keys only.
int fresh_dense_keys(lgc_ctx* ctx, Table* T, int64_t n) {
  if (T->dense && T->cap == n && !T->p) {
    LGC_CUDA_TRY(cudaMemsetAsync(T->bits, 0, sizeof(uint32_t) * ((n + 31) / 32), ctx->stream));
    return LGC_OK;
  }
  table_destroy(ctx, T);
  return table_create_dense(ctx, T, n, false);
}

// Before a round that may add up to `add` keys to a persistent table holding
// `count`: switch to the dense form once it may reach n/8 keys, else grow the
// hashed form to stay at most half full.  Frontier slots are re-resolved.
int ensure_capacity(lgc_ctx* ctx, Table* T, int64_t count, int64_t add, int64_t n,
                    const int32_t* fv, int32_t* fs, int64_t nf) {
  if (T->dense) return LGC_OK;
  const int64_t need = min64(count + add, n);
  if (want_dense(ctx, need, n)) return table_to_dense(ctx, T, n, fv, fs, nf);
  if (2 * need > T->cap) return table_grow(ctx, T, 2 * need, fv, fs, nf);
  return LGC_OK;
}

// Before device-driven rounds: as ensure_capacity for the next round, with
// room ahead (room_slots; a hashed table that would take more memory than the
// dense form becomes dense).
int ensure_room_ahead(lgc_ctx* ctx, Table* T, int64_t count, int64_t add, int64_t n,
                      const int32_t* fv, int32_t* fs, int64_t nf) {
  if (T->dense) return LGC_OK;
  const int64_t need = min64(count + add, n);
  if (want_dense(ctx, need, n) || dense_small(ctx, n)) return table_to_dense(ctx, T, n, fv, fs, nf);
  if (2 * need <= T->cap) return LGC_OK;
  const int64_t cap = room_slots(need, n, 16, kRoomKept);
  if (ctx->table_form == 0 && n >= 1024 && 24 * cap >= 16 * n + n / 8)
    return table_to_dense(ctx, T, n, fv, fs, nf);
  return table_grow(ctx, T, cap, fv, fs, nf);
}

int finish_svec(lgc_ctx* ctx, lgc_graph* g, const Table& T, const double* vals, lgc_svec** p,
                lgc_stats* st_out, lgc_stats& st) {
  int32_t* d_idx = nullptr;
  double* d_val = nullptr;
  int64_t nnz = 0;
  LGC_TRY(table_extract_sorted(ctx, T, vals, g->n, &d_idx, &d_val, &nnz, true, st.touched));
  int s = make_svec(ctx, d_idx, d_val, nnz, ctx->result_on_device, p);
  dfree(ctx, d_idx);
  dfree(ctx, d_val);
  st.table_capacity = T.cap;
  if (st_out) *st_out = st;
  return s;
}

}  // namespace

// Picks the degree bins and the shape of the atomic pull gather for this
// graph: for each light threshold L (vertices of degree <= L one thread each,
// the rest in work items), the lists are rebuilt and every heavy-gather shape
// (edges per lane per batch, lanes per work item, bytes per gathered share)
// gathers a frontier of all vertices into a scratch dense set three times
// after one untimed launch; the light gather of the same share width is
// timed the same way, and the fastest sum of the two medians wins.  The
// gathered sums are exact, so every candidate gives the same values.
int autotune_pull(lgc_ctx* ctx, lgc_graph* g) {
  if (g->n == 0 || g->nnz == 0) return LGC_OK;
  cudaStream_t s = ctx->stream;
  const int64_t n = g->n, words = (n + 31) / 32;
  Table D;
  Fx *shx = nullptr, *hacc = nullptr;
  double* shd = nullptr;
  int32_t *range = nullptr, *hcnt = nullptr, *htouch = nullptr;
  uint32_t* q = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  int st = LGC_OK;
  int gb = 1;
  while (gb < 62 && (int64_t{1} << gb) <= g->max_deg) gb++;
  do {
    if ((st = table_create_dense(ctx, &D, n, false)) || (st = dalloc_t(ctx, &shx, n)) ||
        (st = dalloc_t(ctx, &shd, n)) || (st = dalloc_t(ctx, &range, 2)) ||
        (st = dalloc_t(ctx, &q, words)))
      break;
    if (cudaMemsetAsync(q, 0, 4 * words, s) || cudaEventCreate(&e0) || cudaEventCreate(&e1)) {
      st = LGC_ECUDA;
      break;
    }
    tune_fill_kernel<Fx><<<grid_for(n), kBlock, 0, s>>>(shx, n, range, gb);
    LGC_COUNT_LAUNCH(ctx);
    tune_fill_kernel<double><<<grid_for(n), kBlock, 0, s>>>(shd, n, range, gb);
    LGC_COUNT_LAUNCH(ctx);
    // median of three timed launches after an untimed one
    auto timed = [&](auto&& launch, float* med) {
      float t[3] = {0.f, 0.f, 0.f};
      for (int r = -1; r < 3 && st == LGC_OK; r++) {
        if (cudaEventRecord(e0, s)) st = LGC_ECUDA;
        launch();
        LGC_COUNT_LAUNCH(ctx);
        if (cudaEventRecord(e1, s) || cudaEventSynchronize(e1)) st = LGC_ECUDA;
        if (st == LGC_OK && r >= 0 && cudaEventElapsedTime(&t[r], e0, e1)) st = LGC_ECUDA;
      }
      std::sort(t, t + 3);
      *med = t[1];
    };
    // (batch depth, lanes per item) x (16- or 8-byte shares) x light threshold
    const int cand[7][2] = {{4, 32}, {8, 32}, {16, 32}, {8, 16}, {16, 16}, {8, 8}, {16, 8}};
    const int lights[4] = {32, 64, 128, 256};
    float best_ms = 0.f;
    int best = g->pull_batch, best_group = g->pull_group, best_share = g->pull_share, best_light = g->pull_light;
    bool first = true;
    for (int li = 0; li < 4 && st == LGC_OK; li++) {
      if (g->pull_light != lights[li] && (st = rebuild_pull_lists(ctx, g, lights[li])) != LGC_OK)
        break;
      dfree(ctx, hacc);
      dfree(ctx, hcnt);
      dfree(ctx, htouch);
      hacc = nullptr;
      hcnt = nullptr;
      htouch = nullptr;
      if ((st = dalloc_t(ctx, &hacc, g->nheavy + 1)) ||
          (st = dalloc_t(ctx, &hcnt, g->nheavy + 1)) ||
          (st = dalloc_t(ctx, &htouch, g->nheavy + 1)))
        break;
      if (cudaMemsetAsync(hacc, 0, sizeof(Fx) * (g->nheavy + 1), s) ||
          cudaMemsetAsync(hcnt, 0, 4 * (g->nheavy + 1), s) ||
          cudaMemsetAsync(htouch, 0, 4 * (g->nheavy + 1), s)) {
        st = LGC_ECUDA;
        break;
      }
      const LightView light = g->view(1, g->pull_light);
      for (int sb : {16, 8}) {
        float light_ms = 0.f;
        auto light_of = [&](auto* shv) {
          using SH = std::remove_pointer_t<decltype(shv)>;
          timed([&] {
            pull_light_fx_kernel<SH><<<light_grid(ctx, light), kBlock, 0, s>>>(
                light, shv, range, gb, D, lite_thr(1.0), kFmThreshold, q, ctx->d_counters);
          }, &light_ms);
        };
        if (light.end > light.beg) {
          if (sb == 16) light_of(shx);
          else light_of(shd);
        }
        if (st == LGC_OK && g->nitems == 0 && (first || light_ms < best_ms)) {
          first = false;  // every vertex is light at this threshold
          best_ms = light_ms;
          best_share = sb;
          best_light = lights[li];
        }
        for (int ci = 0; ci < 7 && st == LGC_OK && g->nitems > 0; ci++) {
          const int cb = cand[ci][0], cg = cand[ci][1];
          float med = 0.f;
          auto heavy_of = [&](auto* shv) {
            using SH = std::remove_pointer_t<decltype(shv)>;
            HeavyKernel<SH> heavy = heavy_kernel<SH>(cb, cg);
            const int64_t hb = ceil_div(g->nitems, (kBlock / 32) * (32 / cg));
            const int hg = (int)(hb < (ctx->sms * 16) ? hb : (ctx->sms * 16));
            timed([&] {
              heavy<<<hg, kBlock, 0, s>>>(g->off, g->col, g->items, g->nitems, shv, range, gb, D,
                                          lite_thr(1.0), kFmThreshold, q, hacc, hcnt, htouch,
                                          ctx->d_counters);
            }, &med);
          };
          if (sb == 16) heavy_of(shx);
          else heavy_of(shd);
          if (st != LGC_OK) break;
          if (first || light_ms + med < best_ms) {
            first = false;
            best_ms = light_ms + med;
            best = cb;
            best_group = cg;
            best_share = sb;
            best_light = lights[li];
          }
        }
      }
    }
    if (st == LGC_OK && g->pull_light != best_light)
      st = rebuild_pull_lists(ctx, g, best_light);
    if (st == LGC_OK && !first) {
      g->pull_batch = best;
      g->pull_group = best_group;
      g->pull_share = best_share;
    }
  } while (0);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  table_destroy(ctx, &D);
  for (void* p : {(void*)shx, (void*)shd, (void*)range, (void*)q, (void*)hacc, (void*)hcnt,
                  (void*)htouch})
    dfree(ctx, p);
  cudaMemsetAsync(ctx->d_counters, 0, sizeof(Counters), s);
  if (cudaGetLastError() != cudaSuccess && st == LGC_OK) st = LGC_ECUDA;
  return st;
}

namespace {

// The synchronous PR-Nibble rounds (Sec. 3.3) from the state in W.F, T and
// count until the frontier is empty, or LGC_EMAXROUNDS once max_rounds
// rounds have run in all (W.st.rounds holds the rounds already run).
int prnibble_rounds(lgc_ctx* ctx, lgc_graph* g, PushWork& W, Table& T, int64_t& count,
                    const lgc_prnibble_params* prm, double beta) {
  const double alpha = prm->alpha, eps = prm->eps;
  const bool det = prm->mode == LGC_MODE_DET;
  const double cs = (2.0 * alpha) / (1.0 + alpha);
  const double cn = (1.0 - alpha) / (1.0 + alpha);
  const int64_t max_rounds = prm->max_rounds > 0 ? prm->max_rounds : INT64_MAX;
  int status = LGC_OK;
  lgc_stats& st = W.st;
  while (W.F.size > 0) {
    if (st.rounds >= max_rounds) return LGC_EMAXROUNDS;
    if (rounds_take(ctx, g, W.rmem, W.F.size, W.F.edges, det, beta < 1.0)) {
      // room for the rounds to come: the set grows with them, and a table
      // that fills up costs another launch
      status = ensure_room_ahead(ctx, &T, count, W.F.edges, g->n, W.F.v.ptr, W.F.s.ptr, W.F.size);
      if (status == LGC_ENOMEM) {  // no room ahead: host rounds, which take less
        W.rmem.give_up(ctx);
        continue;
      }
      if (status != LGC_OK) return status;
      status = W.device_rounds_prnibble(T, &count, alpha, cs, cn, eps, prm->rule, det, beta,
                                        max_rounds - st.rounds);
      if (status != LGC_OK) return status;
      continue;
    }
    // room for the round's new keys (at most the frontier's edges)
    if ((status = ensure_capacity(ctx, &T, count, W.F.edges, g->n, W.F.v.ptr, W.F.s.ptr,
                                  W.F.size)) != LGC_OK)
      return status;
    const bool pull = use_pull(ctx, g, W.F.edges);
    if (pull && !T.dense &&
        (status = table_to_dense(ctx, &T, g->n, W.F.v.ptr, W.F.s.ptr, W.F.size)) != LGC_OK)
      return status;
    const bool bulk = use_bulk(det, T, W.F.edges, g->n);
    // beta-fraction rounds: the top ceil(beta |F|) candidates push, the
    // others wait in W.U (after every change of the table's slots)
    if (beta < 1.0 && W.F.size > 1) {
      int64_t m = (int64_t)std::ceil(beta * (double)W.F.size);
      m = std::max<int64_t>(1, std::min<int64_t>(m, W.F.size));
      if (m < W.F.size && (status = W.select_top(T, m)) != LGC_OK) return status;
    }
    W.record_trace();
    const int64_t nf = W.F.size;
    if ((status = W.reserve_frontier_scratch(nf)) != LGC_OK) return status;
    if ((status = W.reserve_next(min64(g->n, count + W.F.edges + nf))) != LGC_OK) return status;
    if ((status = W.reset_counters()) != LGC_OK) return status;
    {
      ProfScope ps(ctx, LGC_PROF_VERTEXMAP, 64.0 * nf);
      vmap_prnibble_kernel<<<vgrid(ctx, nf), kBlock, 0, ctx->stream>>>(
          nf, W.F.v.ptr, W.F.s.ptr, T, g->off, alpha, cs, cn, eps, prm->rule, det ? 1 : 0,
          (!det && !bulk && !pull) ? 1 : 0, W.share.ptr, W.cnt.ptr, W.foff.ptr, W.G.v.ptr,
          W.G.s.ptr, (int32_t)W.G.v.cap, ctx->d_counters);
      LGC_COUNT_LAUNCH(ctx);
    }
    if (cudaGetLastError() != cudaSuccess) {
      return LGC_ECUDA;
    }
    Counters C;
    if (pull) {
      status = W.pull_phase(T, eps, kFmThreshold, &C, det);
    } else {
      int64_t nrec = W.F.edges;
      if (det) {
        // one record per edge and one self record per frontier vertex
        // (cnt[i] = d + 1): the total is known without reading it back
        nrec = W.F.edges + nf;
        if ((status = scan_i64(ctx, W.cnt.ptr, W.epos.ptr, nf, false, W.total.ptr)) != LGC_OK)
          return status;
      } else {
        if ((status = scan_i64(ctx, W.cnt.ptr, W.epos.ptr, nf, false, W.total.ptr)) != LGC_OK)
          return status;
      }
      status = W.edge_phase(T, eps, kFmThreshold, det, true, nrec, &C, bulk);
    }
    if (status != LGC_OK) return status;
    st.rounds++;
    st.pushes += nf;
    st.pushed_edges += W.F.edges;
    count += C.inserted;
    W.G.size = C.next_size;
    W.G.edges = C.next_edges;
    if ((status = W.merge_rest(T, eps)) != LGC_OK) return status;  // candidates that waited
    W.swap_frontiers();
  }
  return status;
}

}  // namespace

// PR-Nibble from the seed set seeds[0..k) with weights (null: all 1) and
// beta-fraction rounds (beta = 1: every candidate pushes).  One seed of
// weight 1 with beta = 1 is Fig. alg:pr-nibble2 / alg:pr-nibble exactly.
int run_prnibble_set(lgc_ctx* ctx, lgc_graph* g, int64_t k, const int32_t* seeds,
                     const double* weights, double beta, const lgc_prnibble_params* prm,
                     lgc_svec** p, lgc_stats* st_out, lgc_svec** r_out) {
  if (!g || k < 1 || !seeds || !prm || !(beta > 0.0 && beta <= 1.0)) return LGC_EINVAL;
  const double alpha = prm->alpha, eps = prm->eps;
  if (!(alpha > 0.0 && alpha < 1.0) || !(eps > 0.0) || (prm->rule != 0 && prm->rule != 1) ||
      (prm->mode != 0 && prm->mode != 1))
    return LGC_EINVAL;
  // r starts as w_i / W (W summed left to right), the seeds in ascending id
  std::vector<std::pair<int32_t, double>> init((size_t)k);
  double Wsum = 0.0;
  int64_t dsum = 0;
  for (int64_t i = 0; i < k; i++) {
    int64_t dx = 0;
    LGC_TRY(validate_seed(ctx, g, seeds[i], &dx));
    const double w = weights ? weights[i] : 1.0;
    if (!(w > 0.0) || !std::isfinite(w)) return LGC_EINVAL;
    Wsum = Wsum + w;
    dsum += dx;
    init[i] = {seeds[i], w};
  }
  for (auto& e : init) e.second = e.second / Wsum;
  std::sort(init.begin(), init.end(),
            [](const std::pair<int32_t, double>& a, const std::pair<int32_t, double>& b) {
              return a.first < b.first;
            });
  for (int64_t i = 1; i < k; i++)
    if (init[i].first == init[i - 1].first) return LGC_EINVAL;  // seeds must be distinct
  ctx->trace_ids.clear();
  ctx->trace_sizes.clear();

  PushWork W(ctx, g);
  Table T;
  // with room ahead for device rounds, without where there is no memory for it
  int made = LGC_ENOMEM;
  if (dense_small(ctx, g->n)) made = table_create_dense(ctx, &T, g->n, true);
  if (made == LGC_ENOMEM && ctx->device_rounds)
    made = table_create(ctx, &T, 2 * std::max<int64_t>(k + dsum, kRoomKeys), true);
  if (made == LGC_ENOMEM) made = table_create(ctx, &T, 2 * (k + dsum), true);
  LGC_TRY(made);
  int64_t count = k;  // keys in T
  int status = LGC_OK;
  int32_t* d_x = nullptr;
  double* d_r = nullptr;
  do {
    if ((status = W.F.v.reserve(ctx, std::max<int64_t>(k, 1024))) != LGC_OK) break;
    if ((status = W.F.s.reserve(ctx, std::max<int64_t>(k, 1024))) != LGC_OK) break;
    if ((status = W.reset_counters()) != LGC_OK) break;
    if (k == 1) {
      init_seed_kernel<<<1, 1, 0, ctx->stream>>>(T, init[0].first, init[0].second, W.F.v.ptr,
                                                  W.F.s.ptr, ctx->d_counters);
    } else {
      std::vector<int32_t> xs((size_t)k);
      std::vector<double> rs((size_t)k);
      for (int64_t i = 0; i < k; i++) {
        xs[i] = init[i].first;
        rs[i] = init[i].second;
      }
      if ((status = dalloc_t(ctx, &d_x, k)) != LGC_OK) break;
      if ((status = dalloc_t(ctx, &d_r, k)) != LGC_OK) break;
      if (cudaMemcpyAsync(d_x, xs.data(), 4 * k, cudaMemcpyHostToDevice, ctx->stream) ||
          cudaMemcpyAsync(d_r, rs.data(), 8 * k, cudaMemcpyHostToDevice, ctx->stream) ||
          cudaStreamSynchronize(ctx->stream)) {  // xs, rs go out of scope
        status = LGC_ECUDA;
        break;
      }
      init_seeds_kernel<<<grid_for(k), kBlock, 0, ctx->stream>>>(T, d_x, d_r, k, W.F.v.ptr,
                                                                  W.F.s.ptr, ctx->d_counters);
    }
    LGC_COUNT_LAUNCH(ctx);
    W.F.size = k;
    W.F.edges = dsum;
    status = prnibble_rounds(ctx, g, W, T, count, prm, beta);
    W.st.touched = count;
  } while (0);
  if (status == LGC_OK || status == LGC_EMAXROUNDS) {
    int s2 = finish_svec(ctx, g, T, T.p, p, st_out, W.st);
    if (s2 == LGC_OK && r_out) {
      // residual of every key (including zeros), for tests
      int32_t* d_idx = nullptr;
      double* d_val = nullptr;
      int64_t nnz = 0;
      s2 = table_extract_sorted(ctx, T, nullptr, g->n, &d_idx, &d_val, &nnz, false);
      if (s2 == LGC_OK) s2 = make_svec(ctx, d_idx, d_val, nnz, false, r_out);
      dfree(ctx, d_idx);
      dfree(ctx, d_val);
    }
    if (s2 != LGC_OK) status = s2;
  }
  table_destroy(ctx, &T);
  dfree(ctx, d_x);
  dfree(ctx, d_r);
  return status;
}

int run_prnibble(lgc_ctx* ctx, lgc_graph* g, int32_t x, const lgc_prnibble_params* prm,
                 lgc_svec** p, lgc_stats* st_out, lgc_svec** r_out) {
  return run_prnibble_set(ctx, g, 1, &x, nullptr, 1.0, prm, p, st_out, r_out);
}

int run_prnibble_from(lgc_ctx* ctx, lgc_graph* g, const Table& src, const int32_t* d_fv,
                      const int32_t* d_fs, int64_t nf, int64_t E, int64_t count,
                      const lgc_prnibble_params* prm, const lgc_stats& so_far, lgc_svec** p,
                      lgc_stats* st_out) {
  if (!src.p || (!src.dense && src.cap < 64) || (src.dense && src.cap != g->n) || nf < 1)
    return LGC_EINVAL;
  cudaStream_t s = ctx->stream;
  PushWork W(ctx, g);
  Table T;
  // the same form and capacity: the same slots
  if (src.dense) LGC_TRY(table_create_dense(ctx, &T, g->n, true));
  else LGC_TRY(table_create(ctx, &T, src.cap, true));
  int status = LGC_OK;
  do {
    const bool copy_ok =
        src.dense
            ? T.dense && cudaMemcpyAsync(T.dval, src.dval, 8 * src.cap, cudaMemcpyDeviceToDevice,
                                         s) == cudaSuccess &&
                  cudaMemcpyAsync(T.bits, src.bits, 4 * ((src.cap + 31) / 32),
                                  cudaMemcpyDeviceToDevice, s) == cudaSuccess &&
                  cudaMemcpyAsync(T.p, src.p, 8 * src.cap, cudaMemcpyDeviceToDevice, s) ==
                      cudaSuccess
            : T.cap == src.cap &&
                  cudaMemcpyAsync(T.s, src.s, sizeof(Slot) * src.cap, cudaMemcpyDeviceToDevice,
                                  s) == cudaSuccess &&
                  cudaMemcpyAsync(T.p, src.p, 8 * src.cap, cudaMemcpyDeviceToDevice, s) ==
                      cudaSuccess;
    if (!copy_ok) {
      status = LGC_ECUDA;
      break;
    }
    if ((status = W.F.v.reserve(ctx, std::max<int64_t>(nf, 1024))) != LGC_OK) break;
    if ((status = W.F.s.reserve(ctx, std::max<int64_t>(nf, 1024))) != LGC_OK) break;
    if (cudaMemcpyAsync(W.F.v.ptr, d_fv, 4 * nf, cudaMemcpyDeviceToDevice, s) ||
        cudaMemcpyAsync(W.F.s.ptr, d_fs, 4 * nf, cudaMemcpyDeviceToDevice, s)) {
      status = LGC_ECUDA;
      break;
    }
    W.F.size = nf;
    W.F.edges = E;
    W.st.rounds = so_far.rounds;
    W.st.pushes = so_far.pushes;
    W.st.pushed_edges = so_far.pushed_edges;
    status = prnibble_rounds(ctx, g, W, T, count, prm, 1.0);
    W.st.touched = count;
  } while (0);
  if (status == LGC_OK || status == LGC_EMAXROUNDS) {
    const int s2 = finish_svec(ctx, g, T, T.p, p, st_out, W.st);
    if (s2 != LGC_OK) status = s2;
    else if (st_out && status == LGC_EMAXROUNDS) st_out->status_detail = LGC_EMAXROUNDS;
  }
  table_destroy(ctx, &T);
  return status == LGC_EMAXROUNDS ? LGC_OK : status;
}

int run_nibble(lgc_ctx* ctx, lgc_graph* g, int32_t x, const lgc_nibble_params* prm, lgc_svec** p,
               lgc_stats* st_out) {
  int64_t dx = 0;
  LGC_TRY(validate_seed(ctx, g, x, &dx));
  const double eps = prm->eps;
  if (prm->T < 0 || !(eps >= 0.0) || (prm->mode != 0 && prm->mode != 1)) return LGC_EINVAL;
  const bool det = prm->mode == LGC_MODE_DET;
  const int fmode = eps > 0.0 ? kFmThreshold : kFmInserted;
  ctx->trace_ids.clear();
  ctx->trace_sizes.clear();

  PushWork W(ctx, g);
  Table Pc, Pn;  // p and p'
  LGC_TRY(table_create(ctx, &Pc, 64, false));
  int64_t count = 1;
  int status = LGC_OK;
  do {
    if ((status = W.F.v.reserve(ctx, 1024)) != LGC_OK) break;
    if ((status = W.F.s.reserve(ctx, 1024)) != LGC_OK) break;
    if ((status = W.reset_counters()) != LGC_OK) break;
    init_seed_kernel<<<1, 1, 0, ctx->stream>>>(Pc, x, 1.0, W.F.v.ptr, W.F.s.ptr, ctx->d_counters);
    LGC_COUNT_LAUNCH(ctx);
    W.F.size = 1;
    W.F.edges = dx;
    lgc_stats& st = W.st;
    for (int t = 1; t <= prm->T; t++) {
      if (rounds_take(ctx, g, W.rmem, W.F.size, W.F.edges, det, false) && (!det || eps > 0.0)) {
        int64_t done = 0;
        bool over = false;
        RoundsFresh q;
        q.eps = eps;
        q.count = count;
        status = W.device_rounds_fresh(Pc, Pn, nullptr, nullptr, &count, q, det, prm->T - t + 1,
                                       &done, &over);
        if (status != LGC_OK || over) break;
        if (done > 0) {
          t += (int)done - 1;  // the loop adds the last one
          continue;
        }
      }
      W.record_trace();
      const int64_t nf = W.F.size;
      const int64_t need = min64(g->n, nf + W.F.edges);
      const bool pull = use_pull(ctx, g, W.F.edges);
      status = pull ? fresh_dense(ctx, &Pn, g->n) : table_fresh(ctx, &Pn, need, g->n, false);
      if (status != LGC_OK) break;  // p' = {}
      const bool bulk = use_bulk(det, Pn, W.F.edges, g->n);
      if ((status = W.reserve_frontier_scratch(nf)) != LGC_OK) break;
      if ((status = W.reserve_next(need)) != LGC_OK) break;
      if ((status = W.reset_counters()) != LGC_OK) break;
      {
        ProfScope ps(ctx, LGC_PROF_VERTEXMAP, 64.0 * nf);
        vmap_nibble_kernel<<<vgrid(ctx, nf), kBlock, 0, ctx->stream>>>(
            nf, W.F.v.ptr, W.F.s.ptr, Pc, Pn, g->off, eps, fmode, det ? 1 : 0,
            (!det && !bulk && !pull) ? 1 : 0, W.share.ptr,
            W.cnt.ptr, W.foff.ptr, W.G.v.ptr, W.G.s.ptr, (int32_t)W.G.v.cap, ctx->d_counters);
        LGC_COUNT_LAUNCH(ctx);
      }
      if (cudaGetLastError() != cudaSuccess) {
        status = LGC_ECUDA;
        break;
      }
      Counters C;
      if (pull) {
        status = W.pull_phase(Pn, eps, fmode, &C, det);
      } else {
        int64_t nrec = W.F.edges;
        if (det) {
          // one record per edge and one self record per frontier vertex
          // (cnt[i] = d + 1): the total is known without reading it back
          nrec = W.F.edges + nf;
          if ((status = scan_i64(ctx, W.cnt.ptr, W.epos.ptr, nf, false, W.total.ptr)) != LGC_OK)
            break;
        } else {
          if ((status = scan_i64(ctx, W.cnt.ptr, W.epos.ptr, nf, false, W.total.ptr)) != LGC_OK)
            break;
        }
        status = W.edge_phase(Pn, eps, fmode, det, true, nrec, &C, bulk);
      }
      if (status != LGC_OK) break;
      st.rounds++;
      st.pushes += nf;
      st.pushed_edges += W.F.edges;
      W.G.size = C.next_size;
      W.G.edges = C.next_edges;
      if (W.G.size == 0) break;  // return the previous p
      std::swap(Pc, Pn);         // p = p'
      count = C.aux + C.inserted;
      W.swap_frontiers();
    }
    st.touched = count;
  } while (0);
  if (status == LGC_OK) status = finish_svec(ctx, g, Pc, nullptr, p, st_out, W.st);
  table_destroy(ctx, &Pc);
  table_destroy(ctx, &Pn);
  return status;
}

int run_hkpr(lgc_ctx* ctx, lgc_graph* g, int32_t x, const lgc_hkpr_params* prm, lgc_svec** p,
             lgc_stats* st_out) {
  int64_t dx = 0;
  LGC_TRY(validate_seed(ctx, g, x, &dx));
  const double t = prm->t, eps = prm->eps;
  const int N = prm->N;
  if (N < 1 || !(t > 0.0) || !(eps >= 0.0) || (prm->mode != 0 && prm->mode != 1))
    return LGC_EINVAL;
  const bool det = prm->mode == LGC_MODE_DET;
  // psi_N = 1, psi_k = 1 + (t/(k+1)) psi_{k+1}; c_j = e^t eps / (2 N psi_j)
  // (the parallel figure's sign of the exponent; LGC_OPT_HK_THRESHOLD_SIGN
  // -1 takes the sequential description's e^-t instead, for comparison)
  std::vector<double> psi(N + 1), c(N + 1);
  psi[N] = 1.0;
  for (int k = N - 1; k >= 0; k--) psi[k] = 1.0 + (t / (double)(k + 1)) * psi[k + 1];
  const double et = ctx->hk_threshold_sign < 0 ? exp(-t) : exp(t);
  for (int j = 0; j <= N; j++) c[j] = (et * eps) / (2.0 * (double)N * psi[j]);
  ctx->trace_ids.clear();
  ctx->trace_sizes.clear();

  PushWork W(ctx, g);
  Table P, Rc, Rn;
  LGC_TRY(table_create(ctx, &P, 2 * (1 + dx), false));
  int status = table_create(ctx, &Rc, 64, false);
  int64_t pcount = 0;
  do {
    if (status != LGC_OK) break;
    if ((status = W.F.v.reserve(ctx, 1024)) != LGC_OK) break;
    if ((status = W.F.s.reserve(ctx, 1024)) != LGC_OK) break;
    if ((status = W.reset_counters()) != LGC_OK) break;
    init_seed_kernel<<<1, 1, 0, ctx->stream>>>(Rc, x, 1.0, W.F.v.ptr, W.F.s.ptr, ctx->d_counters);
    LGC_COUNT_LAUNCH(ctx);
    W.F.size = 1;
    W.F.edges = dx;
    lgc_stats& st = W.st;
    int j = 0;
    while (W.F.size > 0) {
      // (forced pull rounds gather whatever their size, in both modes)
      if (j + 1 < N && ctx->pull_policy != 2 && (!det || eps > 0.0) &&
          rounds_take(ctx, g, W.rmem, W.F.size, W.F.edges, det, false)) {
        status = ensure_room_ahead(ctx, &P, pcount, W.F.size, g->n, nullptr, nullptr, 0);
        if (status == LGC_ENOMEM) {
          W.rmem.give_up(ctx);
          continue;
        }
        if (status != LGC_OK) break;
        int64_t done = 0, rcount = 0;
        bool over = false;
        RoundsFresh q;
        q.t = t;
        q.c = c.data();
        q.N = N;
        q.j = j;
        status = W.device_rounds_fresh(Rc, Rn, &P, &pcount, &rcount, q, det, N - 1 - j, &done,
                                       &over);
        if (status != LGC_OK) break;
        j += (int)done;
        if (done > 0) continue;
      }
      W.record_trace();
      const int64_t nf = W.F.size;
      const bool last = j + 1 >= N;
      // p takes the frontier (and, on the last level, its neighbours)
      if ((status = ensure_capacity(ctx, &P, pcount, nf + (last ? W.F.edges : 0), g->n, nullptr,
                                    nullptr, 0)) != LGC_OK)
        break;
      const bool pull = use_pull(ctx, g, W.F.edges);
      if (pull && last && !P.dense &&
          (status = table_to_dense(ctx, &P, g->n, nullptr, nullptr, 0)) != LGC_OK)
        break;
      if ((status = W.reserve_frontier_scratch(nf)) != LGC_OK) break;
      if ((status = W.reset_counters()) != LGC_OK) break;
      // a pull round of 8-byte shares takes them straight from the vertexMap
      const bool scattered = pull && W.pull_share_bytes(det) == 8;
      if (scattered) {
        if ((status = W.pull_reserve(det)) != LGC_OK) break;
        if (!det && cudaMemsetAsync(W.prange.ptr, 0, 8, ctx->stream) != cudaSuccess) {
          status = LGC_ECUDA;
          break;
        }
        // one reciprocal per degree in place of a division per vertex, where
        // there are more vertices than degrees (b = (j + 1) d is exact and
        // within div_by's range)
        int32_t tab_n =
            nf >= 4 * (int64_t)g->max_deg && j < (1 << 16) ? std::min(g->max_deg + 1, kRecipMax) : 0;
        if (tab_n > 0 && W.recip.reserve(ctx, tab_n) != LGC_OK) tab_n = 0;
        if (tab_n > 0) {
          recip_level_kernel<<<std::min(grid_for(tab_n), 4 * ctx->sms), kBlock, 0, ctx->stream>>>(
              W.recip.ptr, tab_n, last ? 1.0 : (double)(j + 1));
          LGC_COUNT_LAUNCH(ctx);
        }
        // per vertex: fv, fs 8, r 8, degree 4, p read-modify-write 16, share 8
        ProfScope ps(ctx, LGC_PROF_VERTEXMAP, 44.0 * nf);
        vmap_hkpr_pull_kernel<<<vgrid(ctx, nf), kBlock, 0, ctx->stream>>>(
            nf, W.F.v.ptr, W.F.s.ptr, Rc, P, g->deg, t, j, last ? 1 : 0, W.recip.ptr, tab_n,
            W.psh.ptr,
            det ? nullptr : W.prange.ptr, ctx->d_counters);
        LGC_COUNT_LAUNCH(ctx);
      } else {
        ProfScope ps(ctx, LGC_PROF_VERTEXMAP, 64.0 * nf);
        vmap_hkpr_kernel<<<vgrid(ctx, nf), kBlock, 0, ctx->stream>>>(
            nf, W.F.v.ptr, W.F.s.ptr, Rc, P, g->off, t, j, last ? 1 : 0, W.share.ptr, W.cnt.ptr,
            W.foff.ptr, ctx->d_counters);
        LGC_COUNT_LAUNCH(ctx);
      }
      if (cudaGetLastError() != cudaSuccess) {
        status = LGC_ECUDA;
        break;
      }
      if (!pull &&
          (status = scan_i64(ctx, W.cnt.ptr, W.epos.ptr, nf, false, W.total.ptr)) != LGC_OK)
        break;
      Counters C;
      if (!last) {
        const int64_t need = min64(g->n, W.F.edges);
        status = pull ? fresh_dense_keys(ctx, &Rn, g->n)
                      : table_fresh(ctx, &Rn, need, g->n, false);
        if (status != LGC_OK) break;  // r' = {}
        if ((status = W.reserve_next(need)) != LGC_OK) break;
        const double cj = c[j + 1];
        const int fm = cj > 0.0 ? kFmThreshold : kFmInserted;
        if (pull)
          status = W.pull_phase(Rn, cj, fm, &C, det, scattered);
        else
          status = W.edge_phase(Rn, cj, fm, det, false, W.F.edges, &C,
                                use_bulk(det, Rn, W.F.edges, g->n));
        if (status != LGC_OK) break;
        pcount += C.aux;
        st.rounds++;
        st.pushes += nf;
        st.pushed_edges += W.F.edges;
        std::swap(Rc, Rn);  // r = r'
        W.G.size = C.next_size;
        W.G.edges = C.next_edges;
        W.swap_frontiers();
        j++;
      } else {
        if ((status = W.reserve_next(1)) != LGC_OK) break;
        // no frontier after the last level: fire-and-forget adds in either form
        if (pull)
          status = W.pull_phase(P, 0.0, kFmNone, &C, det, scattered);
        else
          status = W.edge_phase(P, 0.0, kFmNone, det, false, W.F.edges, &C, !det);
        if (status != LGC_OK) break;
        pcount += C.aux + C.inserted;
        st.rounds++;
        st.pushes += nf;
        st.pushed_edges += W.F.edges;
        break;
      }
    }
    st.touched = pcount;
  } while (0);
  if (status == LGC_OK) status = finish_svec(ctx, g, P, nullptr, p, st_out, W.st);
  table_destroy(ctx, &P);
  table_destroy(ctx, &Rc);
  table_destroy(ctx, &Rn);
  return status;
}

}  // namespace lgc
