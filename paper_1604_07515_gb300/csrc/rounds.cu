// Consecutive small rounds in one cooperative launch: PR-Nibble's (Sec. 3.3),
// with and without beta-fraction selection, Nibble's (Sec. 3.2) and HK-PR's
// (Sec. 3.4), in atomic and in deterministic mode.
//
// A host-driven round costs its launches and a read-back whatever its size:
// 16 launches and two synchronisations in deterministic mode (records,
// three sort passes, run heads, fold, compaction), 20 with a beta selection
// (three sorts).  On a 60^3 torus (193 rounds of about 3500 vertices) that
// was 125 us a round for work worth a few.  Here a round is a few phases of
// one resident grid separated by grid barriers, and what bounds it is the
// chain of L2 round trips in its phases plus the barriers.
//
// The frontier is an unordered list; every entry carries its vertex, its
// table slot and the position of its first edge in the round's edge list.
// One 64-bit atomic (size << 40 | edges) hands out an entry's list position
// and its edge position together, so no prefix sum is needed before the
// next edge phase.
//
//  atomic mode               V | push |
//  atomic mode, wide rounds  V | exact push | finish |
//  deterministic mode        file | fold and V |
//  beta rounds               first keys | ranks |, and V by itself
//
// V (vertexMap) reads the pushing vertices' r, updates p and r and writes
// their shares.  Atomic mode then adds every edge's share with fetch-and-add
// and appends the vertices an add takes across the threshold.
//
// Wide atomic rounds, those a pull round would take on the host (x_min edges
// or more), keep the pull gather's sums: each destination's shares add up in
// 128-bit fixed point (fx128.cuh; two 64-bit atomics an edge, exact in any
// order) and are rounded once, so the values are those of a pull round, bit
// for bit.
//
// Deterministic mode has to add each destination's contributions in
// ascending source order, whatever order the frontier list is in.  Every
// edge files its pushing entry in its destination's bucket: a destination w
// gets at most d(w) contributions, no two from one source (lgc_graph::
// buckets_fit; other graphs do not come here), so its bucket is the stretch
// [off[w], off[w] + d(w)) of an array as long as the adjacency and needs no
// placing; the returned old count of the destination is the edge's place.
// Then every bucket is put in order and folded by its owner: up to 8
// contributions by one thread (a sorting network in registers), up to 32 by
// a warp (ranks by shuffles), more by a warp or the block through a bitmap
// over the frontier (the order key is then the source's rank among the
// frontier's ids, found by counting) and fold_batch's binade scan.  The sums are the
// sequential fold's, bit for bit.  The owner knows its vertex's final r, so
// it runs the vertex's next V at once (undone where the launch stops before
// the round).  On the torus: 125 us a round host-driven, 20.8 us with the
// buckets counted, placed and scattered in phases and V as another, 13 us
// so (24.4 -> 2.75 ms a call); on a 4096-vertex R-MAT graph, whose hubs get
// about 900 contributions a round, 9.8 -> 2.04 ms a call.
//
// Both modes use that r only grows during an edge phase: the vertices that
// qualify afterwards are those that already did after V (a vertex left
// waiting by the beta selection, or one the original rule leaves at or above
// its threshold) and those a round's contributions take across it.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "edges.cuh"
#include "foldwarp.cuh"
#include "prim.cuh"
#include "rounds.cuh"

namespace cg = cooperative_groups;

namespace lgc {
namespace {

constexpr int kRdBlock = 512;
constexpr int kRdWarps = kRdBlock / 32;
// Rounds taken: at most kRdEdges edges; deterministic ones at most kRdFront
// frontier vertices (the bitmap of a warp, and the quadratic rank count).
constexpr int64_t kRdEdges = int64_t{1} << 20;
constexpr int64_t kRdFront = 16384;
constexpr int64_t kRdRounds = 1024;  // per launch: the host regains control that often
constexpr int kRdShort = 8;          // contributions folded by one thread
constexpr int kRdMid = 128;          // by a warp; more by the block
constexpr int kRdWords = kRdFront / 32;
constexpr int kRdMidWords = 2 * kRdWords + 2 * kRdMid;  // 32-bit words of shared memory per warp
// Shared memory of a deterministic block: the warps' parts, or one bucket's
// bitmap and shares in order.
constexpr int kRdSmemWords = std::max(kRdWarps * kRdMidWords, 2 * kRdWords + 2 * (int)kRdFront);
constexpr int kRdSelf = 1 << 30;     // count of a destination listed before its first edge

// Counters a round adds to.  Round t reads its frontier from set t mod 3 and
// appends to the next; the third is cleared between the round's barriers
// (its last readers are past the first).
struct RdCnt {
  unsigned long long next;      // the round's frontier: size << 40 | degree sum
  unsigned long long push;      // beta rounds: pushing entries, packed alike
  unsigned long long inserted;  // keys created by the round
  unsigned long long pinserted; // HK-PR: keys of p created by it
  int nkeys;                    // fresh sets: entries of the round's key list
  int touched;                  // destinations of the round
  int emin, emax;               // wide rounds: the shares' exponent range, as pull rounds keep it
  int err;
};

// One frontier buffer.
struct RdFront {
  int32_t *v, *s;   // vertex, slot
  uint32_t* e;      // first edge
  int32_t* tile;    // per 32 edges: the entry of their first one
  int32_t* rank;    // deterministic: rank of the entry's id in the frontier
  int32_t* brank;   // beta: rank by (r / d falling, id)
  // deterministic without selection: written by the V of the entry's owner
  double* share;
  int64_t* base;    // off[v] - first edge
  double *r0, *p0;  // r and p before that V
  int4* touched;    // destinations: vertex, slot, first adjacency entry, degree
};

struct RdBuf {
  RdFront F[2];
  unsigned long long* key;  // beta: bits of r / d
  // pushing entries of a V phase (beta: a list of their own)
  int32_t *pv, *pr;         // vertex, rank (beta, deterministic)
  uint32_t* pe;             // first edge (beta)
  int32_t* ptile;           // per 32 edges: the entry of their first one (beta)
  double* share;
  int64_t* base;
  int2* touched;            // wide rounds: destinations
  int32_t* cnt;             // per slot: contributions filed
  Fx* xacc;                 // per slot: a wide round's sum (zero between rounds)
  int32_t* bucket;          // per adjacency entry: pushing entry filed there
  RdCnt* cn;
  int64_t* out;
  int32_t fcap, tiles;      // entries of the frontier arrays, of the tile arrays
};

__device__ inline unsigned long long rd_pack(int64_t size, int64_t edges) {
  return ((unsigned long long)size << 40) | (unsigned long long)edges;
}
__device__ inline int64_t rd_size(unsigned long long p) { return (int64_t)(p >> 40); }
__device__ inline int64_t rd_edges(unsigned long long p) {
  return (int64_t)(p & ((1ull << 40) - 1));
}

// Positions for the lanes with pred in a list counted by *ctr (packed): the
// entry's index, and *epos its first edge.  All lanes of the warp call it.
__device__ inline int64_t rd_take(bool pred, int64_t d, unsigned long long* ctr, uint32_t* epos) {
  const unsigned mask = __ballot_sync(0xffffffffu, pred);
  if (!mask) return -1;
  const int lane = threadIdx.x & 31;
  const int64_t x = pred ? d : 0;
  int64_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  unsigned long long base = 0;
  if (lane == 31) base = atomicAdd(ctr, rd_pack(__popc(mask), inc));
  base = __shfl_sync(0xffffffffu, base, 31);
  *epos = (uint32_t)(rd_edges(base) + inc - x);
  return rd_size(base) + __popc(mask & ((1u << lane) - 1));
}

// Entry `at`, whose edges are [e, e + d), becomes the entry of the 32-edge
// tiles that start among them (every tile start has one writer).
__device__ inline void rd_tiles(int32_t* tile, int32_t tiles, int64_t at, uint32_t e, int64_t d) {
  const int64_t t1 = min((int64_t)tiles, ((int64_t)e + d + 31) / 32);
  for (int64_t t = ((int64_t)e + 31) / 32; t < t1; t++) tile[t] = (int32_t)at;
}

// Appends (v, s) with degree d to frontier F; its position or -1.
__device__ inline int64_t rd_append(const RdBuf& B, const RdFront& F, RdCnt* C, bool pred,
                                    int32_t v, int32_t s, int64_t d, uint32_t* epos) {
  const int64_t pos = rd_take(pred, d, &C->next, epos);
  if (!pred) return -1;
  if (pos >= B.fcap) {
    atomicOr(&C->err, kErrFrontierOverflow);
    return -1;
  }
  F.v[pos] = v;
  F.s[pos] = s;
  F.e[pos] = *epos;
  F.rank[pos] = 0;
  F.brank[pos] = 0;
  rd_tiles(F.tile, B.tiles, pos, *epos, d);
  return pos;
}

// The same by one thread.
__device__ inline void rd_append_one(const RdBuf& B, const RdFront& F, RdCnt* C, int32_t v,
                                     int32_t s, int64_t d) {
  const unsigned long long base = atomicAdd(&C->next, rd_pack(1, d));
  const int64_t pos = rd_size(base);
  const uint32_t e = (uint32_t)rd_edges(base);
  if (pos >= B.fcap) {
    atomicOr(&C->err, kErrFrontierOverflow);
    return;
  }
  F.v[pos] = v;
  F.s[pos] = s;
  F.e[pos] = e;
  F.rank[pos] = 0;
  F.brank[pos] = 0;
  rd_tiles(F.tile, B.tiles, pos, e, d);
}

// Lists the destinations q[k] with k0[k] == 0 (IT per lane, one atomic per
// warp).
template <int IT, class Q>
__device__ inline void rd_touch(Q* list, int* ctr, const Q* q, const int32_t* k0) {
  const int lane = threadIdx.x & 31;
  int mine = 0;
#pragma unroll
  for (int k = 0; k < IT; k++) mine += k0[k] == 0;
  if (!__any_sync(0xffffffffu, mine != 0)) return;
  int inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  int at = 0;
  if (lane == 31) at = atomicAdd(ctr, inc);
  at = __shfl_sync(0xffffffffu, at, 31) + inc - mine;
#pragma unroll
  for (int k = 0; k < IT; k++)
    if (k0[k] == 0) list[at++] = q[k];
}

// The pushing entries of a round: their first edges, edge bases (off[v] -
// first edge) and the tiles' entries.
struct RdEdges {
  const uint32_t* e;
  const int64_t* base;
  const int32_t* tile;
  int64_t np, E;
};

// Every warp takes 32 * IT consecutive edges at a time and calls
// fn(e0, src, at) with each lane's IT edges e0 + 32 k + lane, their pushing
// entries src[k] (-1 past the end) and their places at[k] in the adjacency.
// The first edge's entry comes from the tile array, the others from a window
// of the entries that follow it (edges.cuh).
template <int IT, class Fn>
__device__ inline void rd_edges_of(const RdEdges& R, int64_t warp, int64_t nwarps, Fn&& fn) {
  const int lane = threadIdx.x & 31;
  for (int64_t e0 = warp * 32 * IT; e0 < R.E; e0 += nwarps * 32 * IT) {
    EdgeWindow W(
        R.tile[e0 / 32], R.np, [&](int64_t i) { return (int64_t)R.e[i]; },
        [&](int64_t i) { return R.base[i]; });
    int32_t src[IT];
    int64_t at[IT];
#pragma unroll
    for (int k = 0; k < IT; k++) {
      const int64_t eb = e0 + 32 * k;
      int64_t b = 0;
      const int64_t i = W.find(eb, &b);
      src[k] = eb + lane < R.E ? (int32_t)i : -1;
      at[k] = b + eb + lane;
    }
    fn(e0, src, at);
  }
}

// Where a push's destinations go: a set, the list of the keys a round creates
// in it (fresh sets; null otherwise), and what makes a vertex a candidate: its
// value reaching c * d (thr) or its insertion.
struct RdDest {
  Table T;
  int32_t* keys;
  double c;
  bool thr;
};

// Hot destinations are summed apart (edges.cuh) where the frontier is large
// enough for their adds to queue.  Nibble at eps 1e-7 on 2^22 R-MAT vertices:
// 668 us a call without, 571 with; calls with small frontiers are 2 to 4%
// slower if all rounds do it (PR-Nibble at 1e-6 on 2^18: 190 and 201).  From
// 512 to 8192 makes no difference beyond 2%.
constexpr int64_t kRdHotMin = 2048;

// Atomic push of IT edges a lane: all columns, first probes, slots, adds and
// crossings of a lane's edges side by side.
template <int IT>
__device__ inline void rd_push(const RdBuf& B, const RdDest& D, const HotSet& H,
                               const HotShared& M, bool hot, HotLane<double>& S,
                               const int32_t* __restrict__ col,
                               const int32_t* __restrict__ deg, const RdEdges& R,
                               const RdFront& N, RdCnt* Cc, RdCnt* C, int64_t warp,
                               int64_t nwarps, int64_t* nins) {
  const Table& T = D.T;
  rd_edges_of<IT>(R, warp, nwarps, [&](int64_t, const int32_t* src, const int64_t* at) {
    int32_t w[IT], slot[IT], old_key[IT];
    double sh[IT], old[IT];
    uint32_t probe[IT];
    int ins[IT];
#pragma unroll
    for (int k = 0; k < IT; k++) {
      w[k] = -1;
      sh[k] = 0.0;
      if (src[k] >= 0) {
        w[k] = col[at[k]];
        sh[k] = B.share[src[k]];
      }
    }
    if (hot) hot_take(H, M, S, w, sh);
#pragma unroll
    for (int k = 0; k < IT; k++) {
      probe[k] = 0;
      if (w[k] >= 0)
        probe[k] = T.dense ? __ldcg(&T.bits[w[k] >> 5])
                           : (uint32_t)__ldcg(&T.s[hash_slot(w[k], T.shift)].key);
    }
#pragma unroll
    for (int k = 0; k < IT; k++) {
      slot[k] = -1;
      ins[k] = 0;
      if (w[k] < 0) continue;
      if (T.dense) {
        slot[k] = w[k];
        const uint32_t m = 1u << (w[k] & 31);
        if (!(probe[k] & m) && !(atomicOr(&T.bits[w[k] >> 5], m) & m)) ins[k] = 1;
      } else if ((int32_t)probe[k] == w[k] + 1) {
        slot[k] = (int32_t)hash_slot(w[k], T.shift);
      } else {
        slot[k] = (int32_t)ht_find_or_insert(T, w[k], &ins[k], &Cc->err);
      }
    }
#pragma unroll
    for (int k = 0; k < IT; k++)
      old[k] = slot[k] >= 0 ? atomicAdd(tb_val(T, slot[k]), sh[k]) : 0.0;
#pragma unroll
    for (int k = 0; k < IT; k++) {
      bool pred = false;
      int64_t dw = 0;
      if (slot[k] >= 0) {
        const double nv = old[k] + sh[k];
        if (D.thr ? nv >= D.c : ins[k] != 0) {  // c * d(w) >= c for d(w) >= 1: cheap pre-test
          dw = deg[w[k]];
          const double thr = D.c * (double)dw;
          pred = !D.thr || (old[k] < thr && nv >= thr);
        }
        *nins += ins[k];
      }
      old_key[k] = ins[k] ? 0 : 1;
      uint32_t e;
      rd_append(B, N, C, pred, w[k], slot[k], dw, &e);
    }
    if (D.keys) rd_touch<IT>(D.keys, &Cc->nkeys, slot, old_key);
  });
}

// The hot vertices' sums after a push, each as one add.
__device__ inline void rd_push_hot(const RdBuf& B, const RdDest& D, const HotSet& H,
                                   const HotLane<double>& S, const int32_t* __restrict__ deg,
                                   const RdFront& N, RdCnt* Cc, RdCnt* C, int64_t* nins) {
  const auto join = [](double& a, double x) { a = a + x; };
  hot_flush<kRdWarps>(H, S, join, [&](int32_t w, double sh) {
    int ins = 0;
    const int64_t s = tb_find_or_insert(D.T, w, &ins, &Cc->err);
    if (s < 0) return;
    *nins += ins;
    if (ins && D.keys) D.keys[atomicAdd(&Cc->nkeys, 1)] = (int32_t)s;
    const double old = atomicAdd(tb_val(D.T, s), sh);
    const int64_t d = deg[w];
    const double thr = D.c * (double)d;
    if (D.thr ? old < thr && old + sh >= thr : ins != 0) rd_append_one(B, N, C, w, (int32_t)s, d);
  });
}

// Wide push: every edge's share added to its destination's fixed-point sum;
// a destination's first edge lists it.  Hot destinations are summed apart, as
// in rd_push.
__device__ inline unsigned long long rd_fx_add(Fx* acc, const Fx& x) {
  unsigned long long old = 0;
  if (x.lo) old = atomicAdd((unsigned long long*)&acc->lo, (unsigned long long)x.lo);
  const uint64_t hi = x.hi + (old + x.lo < old ? 1 : 0);
  if (hi) atomicAdd((unsigned long long*)&acc->hi, (unsigned long long)hi);
  return old;
}

template <int IT>
__device__ inline void rd_push_exact(const RdBuf& B, const RdDest& D, const HotSet& H,
                                     const HotShared& M, bool hot, HotLane<Fx>& S,
                                     const int32_t* __restrict__ col,
                                     const RdEdges& R, int L, RdCnt* C, int64_t warp,
                                     int64_t nwarps, int64_t* nins) {
  rd_edges_of<IT>(R, warp, nwarps, [&](int64_t, const int32_t* src, const int64_t* at) {
    int32_t w[IT], slot[IT], k0[IT], old_key[IT];
    Fx x[IT];
    unsigned long long old[IT];
#pragma unroll
    for (int k = 0; k < IT; k++) {
      w[k] = -1;
      x[k] = {0, 0};
      if (src[k] >= 0) {
        w[k] = col[at[k]];
        x[k] = fx_from_bits(fx_bits(B.share[src[k]]), L);
      }
    }
    if (hot)
      hot_take(
          H, M, S, w, x,
          [](const Fx& y, int l) {
            return Fx{__shfl_sync(0xffffffffu, y.lo, l), __shfl_sync(0xffffffffu, y.hi, l)};
          },
          [](Fx& a, const Fx& y) { fx_add(a, y); });
#pragma unroll
    for (int k = 0; k < IT; k++) {
      slot[k] = -1;
      int ins = 0;
      if (w[k] >= 0) slot[k] = (int32_t)tb_find_or_insert(D.T, w[k], &ins, &C->err);
      *nins += ins;
      old_key[k] = ins ? 0 : 1;
    }
#pragma unroll
    for (int k = 0; k < IT; k++) {
      k0[k] = -1;
      old[k] = 0;
      if (slot[k] < 0) continue;
      k0[k] = atomicAdd(&B.cnt[slot[k]], 1);
      if (x[k].lo)
        old[k] = atomicAdd((unsigned long long*)&B.xacc[slot[k]].lo, (unsigned long long)x[k].lo);
    }
#pragma unroll
    for (int k = 0; k < IT; k++) {
      const uint64_t hi = x[k].hi + (old[k] + x[k].lo < old[k] ? 1 : 0);
      if (slot[k] >= 0 && hi)
        atomicAdd((unsigned long long*)&B.xacc[slot[k]].hi, (unsigned long long)hi);
    }
    int2 q[IT];
#pragma unroll
    for (int k = 0; k < IT; k++) q[k] = make_int2(w[k], slot[k]);
    rd_touch<IT>(B.touched, &C->touched, q, k0);
    if (D.keys) rd_touch<IT>(D.keys, &C->nkeys, slot, old_key);
  });
}

__device__ inline void rd_push_exact_hot(const RdBuf& B, const RdDest& D, const HotSet& H,
                                         const HotLane<Fx>& S, RdCnt* C, int64_t* nins) {
  const auto join = [](Fx& a, const Fx& x) { fx_add(a, x); };
  hot_flush<kRdWarps>(H, S, join, [&](int32_t w, const Fx& x) {
    int ins = 0;
    const int64_t s = tb_find_or_insert(D.T, w, &ins, &C->err);
    if (s < 0) return;
    *nins += ins;
    if (ins && D.keys) D.keys[atomicAdd(&C->nkeys, 1)] = (int32_t)s;
    rd_fx_add(&B.xacc[s], x);
    if (atomicAdd(&B.cnt[s], 1) == 0)
      B.touched[atomicAdd(&C->touched, 1)] = make_int2(w, (int32_t)s);
  });
}

// After the barrier: every listed destination's sum joins its value, rounded
// once, as a pull round adds it.
__device__ inline void rd_settle_exact(const RdBuf& B, const RdDest& D,
                                       const int32_t* __restrict__ deg, int L, const RdFront& N,
                                       RdCnt* Cc, RdCnt* C, int64_t warp, int64_t nwarps) {
  const int lane = threadIdx.x & 31;
  const int nt = __ldcg(&Cc->touched);
  for (int64_t b = warp * 32; b < nt; b += nwarps * 32) {
    const int64_t i = b + lane;
    bool pred = false;
    int2 ts = make_int2(0, 0);
    int64_t d = 0;
    if (i < nt) {
      ts = B.touched[i];
      const Fx X = B.xacc[ts.y];
      B.xacc[ts.y] = Fx{0, 0};
      B.cnt[ts.y] = 0;
      double* at = tb_val(D.T, ts.y);
      const double old = *at;
      const double v = old + fx_to_double(X, L);
      *at = v;
      d = deg[ts.x];
      const double thr = D.c * (double)d;
      pred = old < thr && v >= thr;
    }
    uint32_t e;
    rd_append(B, N, C, pred, ts.x, ts.y, d, &e);
  }
}

// Deterministic filing: every edge's pushing entry into its destination's
// bucket; a destination's first edge lists it.
template <int IT>
__device__ inline void rd_file(const RdBuf& B, const Table& T, const int64_t* __restrict__ off,
                               const int32_t* __restrict__ col, const RdEdges& R, int4* touched,
                               int32_t* keys, RdCnt* C, int64_t warp, int64_t nwarps,
                               int64_t* nins) {
  rd_edges_of<IT>(R, warp, nwarps, [&](int64_t, const int32_t* src, const int64_t* at) {
    int32_t slot[IT], k0[IT], old_key[IT];
    int4 q[IT];
#pragma unroll
    for (int k = 0; k < IT; k++) q[k].x = src[k] >= 0 ? col[at[k]] : -1;
#pragma unroll
    for (int k = 0; k < IT; k++) {  // at most kRdEntries entries: 32 bits
      q[k].z = q[k].x >= 0 ? (int32_t)off[q[k].x] : 0;
      q[k].w = q[k].x >= 0 ? (int32_t)off[q[k].x + 1] : 0;
    }
#pragma unroll
    for (int k = 0; k < IT; k++) {
      slot[k] = -1;
      int ins = 0;
      if (q[k].x >= 0) slot[k] = (int32_t)tb_find_or_insert(T, q[k].x, &ins, &C->err);
      *nins += ins;
      old_key[k] = ins ? 0 : 1;
      q[k].y = slot[k];
      q[k].w -= q[k].z;
    }
#pragma unroll
    for (int k = 0; k < IT; k++) k0[k] = slot[k] >= 0 ? atomicAdd(&B.cnt[slot[k]], 1) : -1;
#pragma unroll
    for (int k = 0; k < IT; k++)
      if (slot[k] >= 0) B.bucket[q[k].z + (k0[k] & (kRdSelf - 1))] = src[k];
    rd_touch<IT>(touched, &C->touched, q, k0);
    if (keys) rd_touch<IT>(keys, &C->nkeys, slot, old_key);
  });
}

__device__ inline void rd_cswap(uint32_t& ka, double& a, uint32_t& kb, double& b) {
  const bool s = ka > kb;
  const uint32_t tk = s ? kb : ka;
  const double t = s ? b : a;
  kb = s ? ka : kb;
  b = s ? a : b;
  ka = tk;
  a = t;
}

// What the buckets' entries (pushing entries) stand for.
struct RdSrc {
  const int32_t *id, *rank;  // order by either: the vertex, its rank in the frontier
  const double* share;
};

// A bucket of c <= kRdShort contributions i[0, c) folded into acc in ascending
// id by one thread: Batcher's odd-even merge sort of 8 in registers.
__device__ inline double rd_fold_short(const int32_t i[kRdShort], const RdSrc& S, int c,
                                       double acc) {
  if (c == 0) return acc;
  if (c == 1) return acc + S.share[i[0]];
  uint32_t k[kRdShort];
  double x[kRdShort];
#pragma unroll
  for (int j = 0; j < kRdShort; j++) {
    k[j] = j < c ? (uint32_t)S.id[i[j]] : 0xFFFFFFFFu;
    x[j] = j < c ? S.share[i[j]] : 0.0;
  }
#define LGC_CS(a, b) rd_cswap(k[a], x[a], k[b], x[b])
  LGC_CS(0, 1); LGC_CS(2, 3); LGC_CS(4, 5); LGC_CS(6, 7);
  LGC_CS(0, 2); LGC_CS(1, 3); LGC_CS(4, 6); LGC_CS(5, 7);
  LGC_CS(1, 2); LGC_CS(5, 6);
  LGC_CS(0, 4); LGC_CS(1, 5); LGC_CS(2, 6); LGC_CS(3, 7);
  LGC_CS(2, 4); LGC_CS(3, 5);
  LGC_CS(1, 2); LGC_CS(3, 4); LGC_CS(5, 6);
#undef LGC_CS
#pragma unroll
  for (int j = 0; j < kRdShort; j++)
    if (j < c) acc = acc + x[j];
  return acc;
}

// A bucket of kRdShort < c <= kRdMid contributions, by a warp (acc the same in
// every lane before and after).  sm: kRdMidWords words of the warp's own.
__device__ inline double rd_fold_mid(const int32_t* bucket, const RdSrc& S, int c, int64_t nf,
                                     double acc, uint32_t* sm) {
  const int lane = threadIdx.x & 31;
  double* sorted = reinterpret_cast<double*>(sm + 2 * kRdWords);
  __syncwarp();
  if (c <= 32) {
    const int32_t i = lane < c ? bucket[lane] : -1;
    const uint32_t k = i >= 0 ? (uint32_t)S.id[i] : 0xFFFFFFFFu;
    const double x = i >= 0 ? S.share[i] : 0.0;
    int r = 0;
    for (int j = 0; j < c; j++) r += __shfl_sync(0xffffffffu, k, j) < k ? 1 : 0;
    if (lane < c) sorted[r] = x;
    __syncwarp();
    for (int j = 0; j < c; j++) acc = acc + sorted[j];
    return acc;
  }
  // the ranks are below nf <= kRdFront: a bitmap gives each entry's position
  constexpr int kU = kRdMid / 32;
  uint32_t *bits = sm, *pre = sm + kRdWords;
  const int words = (int)((nf + 31) / 32);
  for (int i = lane; i < words; i += 32) bits[i] = 0;
  int32_t at[kU];
  uint32_t k[kU];
  double x[kU];
#pragma unroll
  for (int j = 0; j < kU; j++) at[j] = 32 * j + lane < c ? bucket[32 * j + lane] : -1;
#pragma unroll
  for (int j = 0; j < kU; j++) {
    k[j] = at[j] >= 0 ? (uint32_t)S.rank[at[j]] : 0u;
    x[j] = at[j] >= 0 ? S.share[at[j]] : 0.0;
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < kU; j++)
    if (at[j] >= 0) atomicOr(&bits[k[j] >> 5], 1u << (k[j] & 31));
  __syncwarp();
  uint32_t run = 0;
  for (int i0 = 0; i0 < words; i0 += 32) {
    const int i = i0 + lane;
    const uint32_t n = i < words ? (uint32_t)__popc(bits[i]) : 0u;
    uint32_t inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (i < words) pre[i] = run + inc - n;
    run += __shfl_sync(0xffffffffu, inc, 31);
  }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < kU; j++)
    if (at[j] >= 0)
      sorted[pre[k[j] >> 5] + __popc(bits[k[j] >> 5] & ((1u << (k[j] & 31)) - 1u))] = x[j];
  __syncwarp();
  // the first contributions by FP64 adds (32 ns each): while the value is
  // small it leaves its binade every few of them, and fold_batch starts again
  // each time
  for (int j = 0; j < 32; j++) acc = acc + sorted[j];
  constexpr int kN = (kRdMid - 32 + 31) / 32;
  double v[kN];
#pragma unroll
  for (int j = 0; j < kN; j++) {
    const int i = 32 + kN * lane + j;
    v[j] = i < c ? sorted[i] : 0.0;  // +0.0 past the end adds nothing
  }
  return fold_batch(acc, v, lane);
}

// fold_batch by the block: folds the kRdBlock shares x (thread t holds
// position t; +0.0 past the list's end) into acc, the same in every thread.
// One share a thread makes a pass over a binade four times shorter than a
// warp's eight a lane.
struct RdFoldMem {
  FoldStep tot[kRdWarps];
  double acc;
  int start;
};
__device__ inline double rd_fold_batch(double acc, double x, RdFoldMem& M) {
  const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  int start = 0;
  while (start < kRdBlock) {  // the same in every thread
    const int bu = fold_binade(acc);
    const int64_t A0 = fold_int(acc);
    const FoldStep st = tid >= start ? fold_step(x, bu) : FoldStep{0, 0};
    const bool par = __syncthreads_or(st.g0 != st.g1) != 0;  // see fold_batch
    FoldStep P = st;  // inclusive over the warp, then over the block
    if (!par) {
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
    // a total of 2^53 or more leaves the binade however large it is: capped,
    // the sums over warps stay in range
    constexpr int64_t kCap = int64_t{1} << 55;
    if (lane == 31) M.tot[wib] = {min(P.g0, kCap), min(P.g1, kCap)};
    if (tid == 0) M.start = kRdBlock;
    __syncthreads();
    FoldStep W = {0, 0};
    if (!par) {
      for (int w = 0; w < wib; w++) W.g0 += M.tot[w].g0;
      W.g1 = W.g0;
    } else {
      for (int w = 0; w < wib; w++) W = fold_compose(W, M.tot[w]);
    }
    const int64_t Aw = fold_apply(W, A0);  // before this warp's shares
    const int64_t A = fold_apply(P, Aw);
    const int64_t up = __shfl_up_sync(0xffffffffu, A, 1);
    const int64_t before = lane ? up : Aw;
    if (A >= kFoldTop && before < kFoldTop) {  // one thread: values only grow
      M.acc = fold_double(before, bu) + x;     // the add that leaves the binade
      M.start = tid + 1;
    } else if (tid == kRdBlock - 1 && A < kFoldTop) {
      M.acc = fold_double(A, bu);
    }
    __syncthreads();
    acc = M.acc;
    start = M.start;
    // the next pass writes M only after its own first barrier
  }
  return acc;
}

// A longer bucket (c <= kRdFront), by the whole block (the result in every
// thread).  sm: the block's kRdSmemWords words.
__device__ inline double rd_fold_block(const int32_t* bucket, const RdSrc& S, int c, int64_t nf,
                                       double acc, uint32_t* sm) {
  __shared__ uint32_t s_tot[kRdWarps];
  __shared__ RdFoldMem s_fold;
  const int tid = threadIdx.x, lane = tid & 31, wib = tid >> 5;
  static_assert(kRdWords == kRdBlock, "one bitmap word per thread");
  uint32_t *bits = sm, *pre = sm + kRdWords;
  double* sorted = reinterpret_cast<double*>(sm + 2 * kRdWords);
  bits[tid] = 0;
  __syncthreads();
  for (int i = tid; i < c; i += kRdBlock) {
    const uint32_t k = (uint32_t)S.rank[bucket[i]];
    atomicOr(&bits[k >> 5], 1u << (k & 31));
  }
  __syncthreads();
  const uint32_t n = (uint32_t)__popc(bits[tid]);
  uint32_t inc = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_tot[wib] = inc;
  __syncthreads();
  uint32_t before = 0;
  for (int w = 0; w < wib; w++) before += s_tot[w];
  pre[tid] = before + inc - n;
  __syncthreads();
  for (int i = tid; i < c; i += kRdBlock) {
    const int32_t e = bucket[i];
    const uint32_t k = (uint32_t)S.rank[e];
    sorted[pre[k >> 5] + __popc(bits[k >> 5] & ((1u << (k & 31)) - 1u))] = S.share[e];
  }
  __syncthreads();
  for (int k0 = 0; k0 < c; k0 += kRdBlock)
    acc = rd_fold_batch(acc, k0 + tid < c ? sorted[k0 + tid] : 0.0, s_fold);
  return acc;
}

// Adds to rank[i] (zero before), for every entry i < nf, the number of
// entries j with before(key j, key i), where get(j) loads a key: tasks of 32
// entries by 32, the keys exchanged by shuffles.
template <class Key, class Get, class Before>
__device__ inline void rd_rank(int64_t nf, int32_t* rank, int64_t warp, int64_t nwarps, Get&& get,
                               Before&& before) {
  const int lane = threadIdx.x & 31;
  const int64_t nb = (nf + 31) / 32;
  for (int64_t t = warp; t < nb * nb; t += nwarps) {
    const int64_t i = (t % nb) * 32 + lane, j = (t / nb) * 32 + lane;
    const int n = (int)min((int64_t)32, nf - (t / nb) * 32);
    const Key mine = get(i < nf ? i : nf - 1), other = get(j < nf ? j : nf - 1);
    int c = 0;
    for (int q = 0; q < n; q++) c += before(other.shfl(q), mine) ? 1 : 0;
    if (i < nf && c) atomicAdd(&rank[i], c);
  }
}

struct RdIdKey {
  int32_t v;
  __device__ RdIdKey shfl(int q) const { return {__shfl_sync(0xffffffffu, v, q)}; }
};
struct RdTopKey {
  unsigned long long k;
  int32_t v;
  __device__ RdTopKey shfl(int q) const {
    return {__shfl_sync(0xffffffffu, k, q), __shfl_sync(0xffffffffu, v, q)};
  }
};

struct RdArgs {
  const int64_t* off;
  const int32_t *col, *deg;
  const int32_t *in_v, *in_s;  // the frontier to start from
  int64_t in_nf;
  double alpha, cs, cn, eps, beta;
  int rule;
  int need_rank;  // a bucket may hold more than 32 contributions
  int gbits;      // sums of fewer than 2^gbits shares
  int keep_room;  // the buffers do not hold every vertex
  int64_t x_min, count, max_rounds, e_max, f_max, key_limit;
  HotSet hot;
};

// The vertexMap's arithmetic for residual r and degree d: the share an edge
// carries, and the residual and the increment of p that stay.
struct RdMapped {
  double share, rbase, dp;
};
__device__ inline RdMapped rd_map(const RdArgs& A, double r, int64_t d) {
  if (A.rule == 0) return {(A.cn * r) / (double)d, 0.0, A.cs * r};
  return {((1.0 - A.alpha) * r) / (2.0 * (double)d), ((1.0 - A.alpha) * r) / 2.0, A.alpha * r};
}

// Why the launch ends before the round with frontier fr (0: it does not).
__device__ inline int rd_stop(const RdArgs& A, const RdBuf& B, unsigned long long fr, int err,
                              int64_t rounds, int64_t count) {
  const int64_t nf = rd_size(fr), E = rd_edges(fr);
  if (err) return 4;
  if (nf == 0) return 1;
  if (rounds >= A.max_rounds) return 2;
  if (E > A.e_max || nf > A.f_max || (A.keep_room && nf + E > B.fcap) || count + E > A.key_limit)
    return 3;
  return 0;
}

__device__ inline void rd_finish(const RdBuf& B, int stop, int err, int cur, unsigned long long fr,
                                 int64_t count, int64_t rounds, int64_t pushes, int64_t pushed) {
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  B.out[0] = stop == 4 ? err : 0;
  B.out[1] = cur;
  B.out[2] = rd_size(fr);
  B.out[3] = rd_edges(fr);
  B.out[4] = count;
  B.out[5] = rounds;
  B.out[6] = pushes;
  B.out[7] = pushed;
}

// The beta selection: ranks of the frontier's entries by (r / d falling,
// ascending id) into F.brank where not all of them push; returns how many
// push.  Ends with a barrier.
__device__ inline int64_t rd_select(const RdArgs& A, const RdBuf& B, const RdFront& F,
                                    const Table& T, int64_t nf, int64_t warp, int64_t nwarps,
                                    cg::grid_group& grid) {
  const int lane = threadIdx.x & 31;
  const int64_t m = max((int64_t)1, min(nf, (int64_t)ceil(A.beta * (double)nf)));
  if (m == nf) return m;
  for (int64_t i = warp * 32 + lane; i < nf; i += nwarps * 32) {
    const double r = F.s[i] >= 0 ? *tb_val(T, F.s[i]) : 0.0;
    B.key[i] = (unsigned long long)__double_as_longlong(r / (double)A.deg[F.v[i]]) &
               0x7FFFFFFFFFFFFFFFull;
  }
  grid.sync();
  rd_rank<RdTopKey>(
      nf, F.brank, warp, nwarps, [&](int64_t i) { return RdTopKey{B.key[i], F.v[i]}; },
      [](const RdTopKey& a, const RdTopKey& b) { return a.k > b.k || (a.k == b.k && a.v < b.v); });
  grid.sync();
  return m;
}

// V over the frontier F as a phase: the pushing entries' p, r, shares and
// edge bases (BETA: in a list of their own), and the vertices that stay
// candidates appended to N.
template <bool DET, bool BETA>
__device__ inline void rd_vmap(const RdArgs& A, const RdBuf& B, const RdFront& F, const RdFront& N,
                               const Table& T, int64_t nf, int64_t m, bool exact, RdCnt* Cc,
                               RdCnt* C, int64_t warp, int64_t nwarps) {
  const int lane = threadIdx.x & 31;
  int emin = 0, emax = 0;
  for (int64_t b = warp * 32; b < nf; b += nwarps * 32) {
    const int64_t i = b + lane;
    bool self = false, push = false;
    int32_t v = 0, s = 0;
    int64_t d = 0, o0 = 0;
    double sh = 0.0;
    if (i < nf) {
      v = F.v[i];
      s = F.s[i];
      const bool ok = s >= 0;
      push = !BETA || m == nf || F.brank[i] < m;
      double r = ok ? *tb_val(T, s) : 0.0;
      o0 = A.off[v];
      d = A.off[v + 1] - o0;
      if (push) {
        const RdMapped q = rd_map(A, r, d);
        if (ok) {
          T.p[s] = T.p[s] + q.dp;
          *tb_val(T, s) = q.rbase;
        }
        r = q.rbase;
        sh = q.share;
        if (exact && sh > 0.0) {
          const int be = fx_bexp(fx_bits(sh));
          emin = max(emin, 2047 - be);
          emax = max(emax, be);
        }
        if (!BETA) {
          B.share[i] = sh;
          B.base[i] = o0 - (int64_t)F.e[i];
        }
      }
      self = ok && (!push || A.rule == 1) && r >= A.eps * (double)d;
    }
    if (BETA) {
      uint32_t e;
      const int64_t at = rd_take(push, d, &Cc->push, &e);
      if (push) {
        B.pe[at] = e;
        B.share[at] = sh;
        B.base[at] = o0 - (int64_t)e;
        rd_tiles(B.ptile, B.tiles, at, e, d);
        if (DET) {
          B.pv[at] = v;
          B.pr[at] = F.rank[i];
        }
      }
    }
    uint32_t e;
    rd_append(B, N, C, self, v, s, d, &e);
  }
  if (exact) {
    emin = __reduce_max_sync(0xffffffffu, emin);
    emax = __reduce_max_sync(0xffffffffu, emax);
    if (lane == 0 && (emin | emax)) {
      atomicMax(&Cc->emin, emin);
      atomicMax(&Cc->emax, emax);
    }
  }
}

__device__ inline void rd_count_inserted(int64_t nins, RdCnt* C) {
  for (int o = 16; o > 0; o >>= 1) nins += __shfl_xor_sync(0xffffffffu, nins, o);
  if ((threadIdx.x & 31) == 0 && nins)
    atomicAdd(&C->inserted, (unsigned long long)nins);
}

// The edge phase of an atomic round over the edges R: the push, and for a
// wide round (exact) the barrier and the sums' settling.
__device__ inline void rd_push_round(const RdBuf& B, const RdDest& D, const HotSet& H,
                                     const HotShared& M,
                                     const int32_t* __restrict__ col,
                                     const int32_t* __restrict__ deg, const RdEdges& R, bool exact,
                                     int gbits, const RdFront& N, RdCnt* Cc, RdCnt* C,
                                     int64_t warp, int64_t nwarps, cg::grid_group& grid) {
  int64_t nins = 0;
  const bool wide = R.E > nwarps * 64;  // several edges a lane once every warp has work
  const bool hot = H.tab && R.np >= kRdHotMin;
  if (exact) {
    HotLane<Fx> S;
    const int L = fx_scale(2047 - __ldcg(&Cc->emin), __ldcg(&Cc->emax), gbits);
    if (wide) rd_push_exact<4>(B, D, H, M, hot, S, col, R, L, Cc, warp, nwarps, &nins);
    else rd_push_exact<1>(B, D, H, M, hot, S, col, R, L, Cc, warp, nwarps, &nins);
    if (hot) rd_push_exact_hot(B, D, H, S, Cc, &nins);
    rd_count_inserted(nins, Cc);
    grid.sync();
    rd_settle_exact(B, D, deg, L, N, Cc, C, warp, nwarps);
  } else {
    HotLane<double> S;
    if (wide) rd_push<4>(B, D, H, M, hot, S, col, deg, R, N, Cc, C, warp, nwarps, &nins);
    else rd_push<1>(B, D, H, M, hot, S, col, deg, R, N, Cc, C, warp, nwarps, &nins);
    if (hot) rd_push_hot(B, D, H, S, deg, N, Cc, C, &nins);
    rd_count_inserted(nins, Cc);
  }
}

// Atomic mode.
template <bool BETA>
__global__ void __launch_bounds__(kRdBlock, 1) rounds_kernel(RdArgs A, RdBuf B, Table T) {
  __shared__ HotShared s_tab;
  hot_load(A.hot, s_tab);
  cg::grid_group grid = cg::this_grid();
  const int lane = threadIdx.x & 31;
  // consecutive warps on different SMs: a small phase spreads over the chip
  const int64_t warp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int64_t nwarps = (int64_t)gridDim.x * kRdWarps;
  int64_t rounds = 0, pushes = 0, pushed = 0, count = A.count;
  int err = 0;
  for (int64_t b = warp * 32; b < A.in_nf; b += nwarps * 32) {
    const int64_t i = b + lane;
    const bool ok = i < A.in_nf;
    const int32_t v = ok ? A.in_v[i] : 0;
    uint32_t e;
    rd_append(B, B.F[0], &B.cn[0], ok, v, ok ? A.in_s[i] : 0, ok ? A.deg[v] : 0, &e);
  }
  grid.sync();
  for (int set = 0;; set = set == 2 ? 0 : set + 1) {
    const int cur = (int)(rounds & 1);
    RdCnt *Cc = &B.cn[set], *C = &B.cn[set == 2 ? 0 : set + 1];
    RdCnt* Cz = &B.cn[set == 0 ? 2 : set - 1];
    const RdFront &F = B.F[cur], &N = B.F[cur ^ 1];
    const unsigned long long fr = __ldcg(&Cc->next);
    err |= __ldcg(&Cc->err);
    const int stop = rd_stop(A, B, fr, err, rounds, count);
    if (stop) {  // the same decision in every thread: no barrier is left waiting
      rd_finish(B, stop, err, cur, fr, count, rounds, pushes, pushed);
      return;
    }
    const int64_t nf = rd_size(fr), E = rd_edges(fr);
    const bool exact = E >= A.x_min;
    const int64_t m = BETA ? rd_select(A, B, F, T, nf, warp, nwarps, grid) : nf;
    rd_vmap<false, BETA>(A, B, F, N, T, nf, m, exact, Cc, C, warp, nwarps);
    grid.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) *Cz = RdCnt{};
    const unsigned long long pp = BETA ? __ldcg(&Cc->push) : fr;
    const int64_t np = rd_size(pp), Ep = rd_edges(pp);
    const RdEdges R = {BETA ? B.pe : F.e, B.base, BETA ? B.ptile : F.tile, np, Ep};
    const RdDest D = {T, nullptr, A.eps, true};
    rd_push_round(B, D, A.hot, s_tab, A.col, A.deg, R, exact, A.gbits, N, Cc, C, warp, nwarps, grid);
    grid.sync();
    rounds += 1;
    pushes += np;
    pushed += Ep;
    count += (int64_t)__ldcg(&Cc->inserted);
    err |= __ldcg(&Cc->err);
  }
}

// The fold phase of a deterministic round: every listed destination's bucket
// folded into its value; settle(ok, destination, value before, value after, p)
// is then called by whole warps.  Block b takes destinations b, b + gridDim.x,
// ... (the first ones listed are the hubs), a thread each; longer buckets are
// left to the warps, the longest to the block.
template <class Settle>
__device__ inline void rd_fold(const RdBuf& B, const Table& T, const RdSrc& S, const int4* touched,
                               int64_t nf, RdCnt* Cc, uint32_t* s_mem, bool want_p,
                               Settle&& settle) {
  // the block's buckets for a warp and for the block: thread and count; per
  // thread the bucket's place, the value before and the one after
  __shared__ int2 s_mid[kRdBlock], s_big[kRdBlock];
  __shared__ int s_n[2];
  __shared__ int32_t s_o[kRdBlock];
  __shared__ double s_val[kRdBlock];
  const int lane = threadIdx.x & 31;
  uint32_t* sm = s_mem + (threadIdx.x >> 5) * kRdMidWords;
  const int nt = __ldcg(&Cc->touched);
  const int64_t mine = (nt - (int64_t)blockIdx.x + gridDim.x - 1) / gridDim.x;  // <= 0: none
  for (int64_t j0 = 0; j0 < mine; j0 += kRdBlock) {
    if (threadIdx.x < 2) s_n[threadIdx.x] = 0;
    __syncthreads();
    const int64_t j = j0 + threadIdx.x;
    const bool ok = j < mine;
    int4 ts = make_int4(0, 0, 0, 0);
    int c = 0;
    double old = 0.0, acc = 0.0, p = 0.0;
    if (ok) {
      // everything a destination needs next, at once: its count, its values
      // and the first entries of its bucket
      ts = touched[j * gridDim.x + blockIdx.x];
      c = B.cnt[ts.y] & (kRdSelf - 1);
      old = *tb_val(T, ts.y);
      if (want_p) p = T.p[ts.y];
      int32_t q[kRdShort];
#pragma unroll
      for (int k = 0; k < kRdShort; k++) q[k] = k < ts.w ? B.bucket[ts.z + k] : 0;
      B.cnt[ts.y] = 0;
      if (c > kRdShort) {
        const int big = c > kRdMid ? 1 : 0;
        (big ? s_big : s_mid)[atomicAdd(&s_n[big], 1)] = make_int2(threadIdx.x, c);
        s_o[threadIdx.x] = ts.z;
        s_val[threadIdx.x] = old;
      } else {
        acc = rd_fold_short(q, S, c, old);
      }
    }
    __syncthreads();
    const int nmid = s_n[0], nbig = s_n[1];
    for (int k = threadIdx.x >> 5; k < nmid; k += kRdWarps) {
      const int2 q = s_mid[k];
      const double x = rd_fold_mid(B.bucket + s_o[q.x], S, q.y, nf, s_val[q.x], sm);
      if (lane == 0) s_val[q.x] = x;
    }
    for (int k = 0; k < nbig; k++) {
      __syncthreads();  // the shared memory of the buckets before
      const int2 q = s_big[k];
      const double x = rd_fold_block(B.bucket + s_o[q.x], S, q.y, nf, s_val[q.x], s_mem);
      if (threadIdx.x == 0) s_val[q.x] = x;
    }
    __syncthreads();
    if (j - lane < mine) {  // uniform in the warp
      if (c > kRdShort) acc = s_val[threadIdx.x];
      if (ok) *tb_val(T, ts.y) = acc;
      settle(ok, ts, old, acc, p);
    }
  }
}

// Deterministic mode.
template <bool BETA>
__global__ void __launch_bounds__(kRdBlock, 1) rounds_det_kernel(RdArgs A, RdBuf B, Table T) {
  extern __shared__ uint32_t s_mem[];
  cg::grid_group grid = cg::this_grid();
  const int lane = threadIdx.x & 31;
  const int64_t warp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int64_t nwarps = (int64_t)gridDim.x * kRdWarps;
  int64_t rounds = 0, pushes = 0, pushed = 0, count = A.count;
  int err = 0;
  // The vertices with pred (residual r, p, adjacency [o, o + d)) join frontier
  // N of counters C: by themselves with a selection to come, else with their
  // V done.
  auto enter = [&](const RdFront& N, RdCnt* C, bool pred, int32_t v, int32_t s, int64_t o,
                   int64_t d, double r, double p) {
    uint32_t e;
    const int64_t at = rd_append(B, N, C, pred, v, s, d, &e);
    if (BETA) return;
    int32_t k0 = 1;
    if (at >= 0) {
      const RdMapped q = rd_map(A, r, d);
      N.r0[at] = r;
      N.p0[at] = p;
      T.p[s] = p + q.dp;
      *tb_val(T, s) = q.rbase;
      N.share[at] = q.share;
      N.base[at] = o - (int64_t)e;
      if (A.rule == 1 && q.rbase >= A.eps * (double)d) {  // a candidate without contributions too
        B.cnt[s] = kRdSelf;
        k0 = 0;
      }
    }
    const int4 q = make_int4(v, s, (int32_t)o, (int32_t)d);
    if (A.rule == 1) rd_touch<1>(N.touched, &C->touched, &q, &k0);
  };
  for (int64_t b = warp * 32; b < A.in_nf; b += nwarps * 32) {
    const int64_t i = b + lane;
    const bool ok = i < A.in_nf;
    const int32_t v = ok ? A.in_v[i] : 0, s = ok ? A.in_s[i] : 0;
    const int64_t o = ok ? A.off[v] : 0;
    enter(B.F[0], &B.cn[0], ok, v, s, o, ok ? A.off[v + 1] - o : 0, ok ? *tb_val(T, s) : 0.0,
          ok ? T.p[s] : 0.0);
  }
  grid.sync();
  for (int set = 0;; set = set == 2 ? 0 : set + 1) {
    const int cur = (int)(rounds & 1);
    RdCnt *Cc = &B.cn[set], *C = &B.cn[set == 2 ? 0 : set + 1];
    RdCnt* Cz = &B.cn[set == 0 ? 2 : set - 1];
    const RdFront &F = B.F[cur], &N = B.F[cur ^ 1];
    const unsigned long long fr = __ldcg(&Cc->next);
    err |= __ldcg(&Cc->err);
    const int64_t nf = rd_size(fr);
    const int stop = rd_stop(A, B, fr, err, rounds, count);
    if (stop) {  // the same decision in every thread: no barrier is left waiting
      if (!BETA && stop != 4) {  // the V of a round that is not run
        for (int64_t i = warp * 32 + lane; i < nf; i += nwarps * 32) {
          const int32_t s = F.s[i];
          *tb_val(T, s) = F.r0[i];
          T.p[s] = F.p0[i];
          B.cnt[s] = 0;
        }
      }
      rd_finish(B, stop, err, cur, fr, count, rounds, pushes, pushed);
      return;
    }
    // the ranks of the frontier's ids, for buckets too long for shuffles
    if (A.need_rank)
      rd_rank<RdIdKey>(
          nf, F.rank, warp, nwarps, [&](int64_t i) { return RdIdKey{F.v[i]}; },
          [](const RdIdKey& a, const RdIdKey& b) { return a.v < b.v; });
    if (BETA) {
      const int64_t m = rd_select(A, B, F, T, nf, warp, nwarps, grid);
      if (m == nf) grid.sync();  // the ranks are read next
      rd_vmap<true, true>(A, B, F, N, T, nf, m, false, Cc, C, warp, nwarps);
      grid.sync();
    }
    const unsigned long long pp = BETA ? __ldcg(&Cc->push) : fr;
    const int64_t np = rd_size(pp), Ep = rd_edges(pp);
    const RdEdges R = {BETA ? B.pe : F.e, BETA ? B.base : F.base, BETA ? B.ptile : F.tile, np, Ep};
    int64_t nins = 0;
    if (Ep > nwarps * 64)  // several edges a lane once every warp has work
      rd_file<4>(B, T, A.off, A.col, R, F.touched, nullptr, Cc, warp, nwarps, &nins);
    else
      rd_file<1>(B, T, A.off, A.col, R, F.touched, nullptr, Cc, warp, nwarps, &nins);
    rd_count_inserted(nins, Cc);
    grid.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) *Cz = RdCnt{};
    const RdSrc S = BETA ? RdSrc{B.pv, B.pr, B.share} : RdSrc{F.v, F.rank, F.share};
    // p of the destinations, for those that enter
    rd_fold(B, T, S, F.touched, nf, Cc, s_mem, !BETA, [&](bool ok, int4 ts, double old, double acc,
                                                         double p) {
      const double thr = A.eps * (double)ts.w;
      // with a selection the waiting and kept candidates are listed already
      enter(N, C, ok && acc >= thr && (!BETA || old < thr), ts.x, ts.y, ts.z, ts.w, acc, p);
    });
    grid.sync();
    rounds += 1;
    pushes += np;
    pushed += Ep;
    count += (int64_t)__ldcg(&Cc->inserted);
    err |= __ldcg(&Cc->err);
  }
}

// Rounds into fresh sets: Nibble (KIND 0: p'[v] = p[v]/2 on the frontier and
// share p[v]/(2 d)) and HK-PR (KIND 1: p[v] += r[v] and share
// t r[v]/((j+1) d), r' fresh).  The new set of round k is T[k mod 3], its
// source T[(k-1) mod 3] (T[3] in the first round); the third one, the source
// of the round before (still the result where a Nibble round's frontier comes
// out empty), is cleared by its list of keys, so a round costs what it
// touches.  V | push | (wide rounds: settle |), or V | file | fold |: what a
// round takes is a dozen us; with prefix sums for the edges, tables cleared
// in full and every hub's adds queueing it was 52 (13 rounds of a scale-22
// Nibble).
struct RfArgs {
  double t;
  const double* c;  // thresholds by level (device)
  int N, j0;
  int64_t pcount, p_limit;
};
struct RfTabs {
  Table T[4], P;
  int32_t* keys[3];
};

template <bool DET, int KIND>
__global__ void __launch_bounds__(kRdBlock, 1)
    rounds_fresh_kernel(RdArgs A, RfArgs X, RdBuf B, RfTabs Q) {
  extern __shared__ uint32_t s_mem[];
  __shared__ HotShared s_tab;
  if (!DET) hot_load(A.hot, s_tab);
  cg::grid_group grid = cg::this_grid();
  const int lane = threadIdx.x & 31;
  const int64_t warp = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int64_t nwarps = (int64_t)gridDim.x * kRdWarps;
  int64_t rounds = 0, pushes = 0, pushed = 0, pcount = X.pcount;
  int64_t count = A.count, before = A.count;  // keys of the newest set, of its source
  int nk[3] = {0, 0, 0};                      // keys listed per table
  int err = 0;
  for (int64_t b = warp * 32; b < A.in_nf; b += nwarps * 32) {
    const int64_t i = b + lane;
    const bool ok = i < A.in_nf;
    const int32_t v = ok ? A.in_v[i] : 0;
    uint32_t e;
    rd_append(B, B.F[0], &B.cn[0], ok, v, ok ? A.in_s[i] : 0, ok ? A.deg[v] : 0, &e);
  }
  grid.sync();
  for (int set = 0;; set = set == 2 ? 0 : set + 1) {
    const int cur = (int)(rounds & 1);
    RdCnt *Cc = &B.cn[set], *C = &B.cn[set == 2 ? 0 : set + 1];
    RdCnt* Cz = &B.cn[set == 0 ? 2 : set - 1];
    const RdFront &F = B.F[cur], &N = B.F[cur ^ 1];
    // round k uses set k mod 3 and table k mod 3: the same index
    const int src = rounds == 0 ? 3 : (set == 0 ? 2 : set - 1), old = set == 2 ? 0 : set + 1;
    const unsigned long long fr = __ldcg(&Cc->next);
    err |= __ldcg(&Cc->err);
    const int64_t nf = rd_size(fr), E = rd_edges(fr);
    const int j = X.j0 + (int)rounds;
    int stop = 0;
    if (err) stop = 4;
    else if (nf == 0) stop = 1;
    else if (rounds >= A.max_rounds || (KIND == 1 && j + 1 >= X.N)) stop = 2;
    else if (E > A.e_max || nf > A.f_max || (A.keep_room && nf + E > B.fcap) ||
             nf + E > A.key_limit || (KIND == 1 && pcount + nf > X.p_limit))
      stop = 3;
    if (stop) {  // the same decision in every thread: no barrier is left waiting
      rd_finish(B, stop, err, cur, fr, count, rounds, pushes, pushed);
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        // an empty Nibble frontier: the vector before the round that made it
        const bool back = KIND == 0 && stop == 1;
        B.out[4] = back ? before : count;
        B.out[8] = !back ? src : rounds <= 1 ? 3 : old;
        B.out[9] = pcount;
      }
      return;
    }
    const Table S = Q.T[src], D = Q.T[set];
    const double c = KIND == 0 ? A.eps : X.c[j + 1];
    const bool thr = c > 0.0;
    const bool exact = !DET && thr && E >= A.x_min;
    // the ranks of the frontier's ids, for buckets too long for shuffles
    if (DET && A.need_rank)
      rd_rank<RdIdKey>(
          nf, F.rank, warp, nwarps, [&](int64_t i) { return RdIdKey{F.v[i]}; },
          [](const RdIdKey& a, const RdIdKey& b) { return a.v < b.v; });
    // V
    int64_t nins = 0, pins = 0;
    int emin = 0, emax = 0;
    for (int64_t b = warp * 32; b < nf; b += nwarps * 32) {
      const int64_t i = b + lane;
      bool self = false;
      int32_t v = 0, ds = 0, k0 = 1;
      int64_t d = 0;
      if (i < nf) {
        v = F.v[i];
        const int32_t s = F.s[i];
        const double r = s >= 0 ? *tb_val(S, s) : 0.0;
        const int64_t o0 = A.off[v];
        d = A.off[v + 1] - o0;
        double sh;
        if (KIND == 0) {
          int ins = 0;
          ds = (int32_t)tb_find_or_insert(D, v, &ins, &Cc->err);
          const double half = r / 2.0;
          if (ds >= 0) *tb_val(D, ds) = half;
          nins += ins;
          k0 = ins ? 0 : 1;
          sh = r / (2.0 * (double)d);
          self = ds >= 0 && (!thr || half >= c * (double)d);
        } else {
          int ins = 0;
          const int64_t ps = tb_find_or_insert(Q.P, v, &ins, &Cc->err);
          if (ps >= 0) *tb_val(Q.P, ps) = *tb_val(Q.P, ps) + r;
          pins += ins;
          sh = (X.t * r) / ((double)(j + 1) * (double)d);
        }
        if (exact && sh > 0.0) {
          const int be = fx_bexp(fx_bits(sh));
          emin = max(emin, 2047 - be);
          emax = max(emax, be);
        }
        B.share[i] = sh;
        B.base[i] = o0 - (int64_t)F.e[i];
      }
      if (KIND == 0) {
        rd_touch<1>(Q.keys[set], &Cc->nkeys, &ds, &k0);
        uint32_t e;
        rd_append(B, N, C, self, v, ds, d, &e);
      }
    }
    if (exact) {
      emin = __reduce_max_sync(0xffffffffu, emin);
      emax = __reduce_max_sync(0xffffffffu, emax);
      if (lane == 0 && (emin | emax)) {
        atomicMax(&Cc->emin, emin);
        atomicMax(&Cc->emax, emax);
      }
    }
    if (KIND == 1) {
      for (int o = 16; o > 0; o >>= 1) pins += __shfl_xor_sync(0xffffffffu, pins, o);
      if (lane == 0 && pins) atomicAdd(&Cc->pinserted, (unsigned long long)pins);
    }
    // the table after next, by its keys
    for (int64_t i = warp * 32 + lane; i < nk[old]; i += nwarps * 32) {
      const int32_t k = Q.keys[old][i];
      const Table& Z = Q.T[old];
      if (Z.dense) {
        Z.dval[k] = 0.0;
        Z.bits[k >> 5] = 0;  // every key of the word goes
      } else {
        Z.s[k] = Slot{};
      }
    }
    rd_count_inserted(nins, Cc);
    grid.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) *Cz = RdCnt{};
    const RdEdges R = {F.e, B.base, F.tile, nf, E};
    if (DET) {
      int64_t fins = 0;
      if (E > nwarps * 64)
        rd_file<4>(B, D, A.off, A.col, R, F.touched, Q.keys[set], Cc, warp, nwarps, &fins);
      else
        rd_file<1>(B, D, A.off, A.col, R, F.touched, Q.keys[set], Cc, warp, nwarps, &fins);
      rd_count_inserted(fins, Cc);
      grid.sync();
      rd_fold(B, D, RdSrc{F.v, F.rank, B.share}, F.touched, nf, Cc, s_mem, false,
              [&](bool ok, int4 ts, double old_v, double acc, double) {
                // a level without a threshold takes every key the round
                // created: in HK-PR's empty set, every destination
                const double th = c * (double)ts.w;
                uint32_t e;
                rd_append(B, N, C, ok && (!thr || (old_v < th && acc >= th)), ts.x, ts.y, ts.w,
                          &e);
              });
    } else {
      const RdDest dest = {D, Q.keys[set], c, thr};
      rd_push_round(B, dest, A.hot, s_tab, A.col, A.deg, R, exact, A.gbits, N, Cc, C, warp, nwarps,
                    grid);
    }
    grid.sync();
    rounds += 1;
    pushes += nf;
    pushed += E;
    before = count;
    nk[set] = __ldcg(&Cc->nkeys);
    nk[old] = 0;
    count = nk[set];
    pcount += (int64_t)__ldcg(&Cc->pinserted);
    err |= __ldcg(&Cc->err);
  }
}

using RdKernel = void (*)(RdArgs, RdBuf, Table);

// The rounds' edge limit on this graph.
int64_t rd_emax(const lgc_graph* g) { return std::min<int64_t>(kRdEdges, g->nnz); }
// Buckets of more than 32 contributions are ordered by rank.
bool rd_ranks(const lgc_graph* g) { return g->max_deg > 32; }

}  // namespace

bool rounds_take(const lgc_ctx* ctx, const lgc_graph* g, const RoundsMem& M, int64_t nf, int64_t E,
                 bool det, bool beta) {
  // (EdgeWindow: every source has edges)
  if (!ctx->device_rounds || ctx->trace || nf <= 0 || E > rd_emax(g) || g->sinks || M.no_room)
    return false;
  if (det) {
    // every deterministic round is to gather, or lists that could overflow the
    // buckets
    if (ctx->pull_policy == 2 || !g->buckets_fit || g->nnz > kRdEntries) return false;
    if (rd_ranks(g) && nf > kRdFront) return false;
  }
  return !beta || nf <= kRdFront;
}

namespace {

// What a launch is given: limits, buffers carved from M's slab, arguments.
struct RdLaunch {
  RdArgs A{};
  RdBuf B{};
};

// fresh_keys: room for the key lists of fresh sets (else null); levels: room
// for that many thresholds (device) in *levels.  *no_room: M has given up.
int rd_prepare(lgc_ctx* ctx, lgc_graph* g, RoundsMem& M, int64_t slots, const int32_t* fv,
               const int32_t* fs, int64_t nf, bool det, bool sel, bool staged, int64_t x_min,
               int64_t max_rounds, int64_t key_limit, int32_t** fresh_keys, int64_t levels,
               double** level_c, RdLaunch* L, bool* no_room) {
  cudaStream_t s = ctx->stream;
  RdBuf& B = L->B;
  RdArgs& A = L->A;
  *no_room = false;
  const bool wide = !det && x_min <= rd_emax(g);  // wide rounds may occur
  const int64_t e_max = rd_emax(g);
  // a next frontier has at most nf + E entries, all distinct
  const int64_t fcap = std::min<int64_t>(g->n, 2 * kRdEdges);
  const int64_t f_max = sel || (det && rd_ranks(g)) ? std::min<int64_t>(kRdFront, fcap) : fcap;
  // without room for all of it the rounds stay on the host
  auto take = [&](auto** p, size_t count) {
    const int st = dalloc_t(ctx, p, count);
    if (st == LGC_ENOMEM) {
      M.give_up(ctx);
      *no_room = true;
    }
    return st;
  };
  if (det && !M.bucket) {
    const int st = take(&M.bucket, (size_t)g->nnz);
    if (st != LGC_OK) return *no_room ? LGC_OK : st;
  }
  const int64_t tiles = e_max / 32 + 1;
  // carve one slab; staged: a V phase writes the shares (else the entries' owners)
  size_t at = 0;
  char* base = nullptr;
  auto carve = [&](auto** p, int64_t n, bool want) {
    using P = std::remove_pointer_t<std::remove_pointer_t<decltype(p)>>;
    *p = want ? reinterpret_cast<P*>(base + at) : nullptr;
    if (want) at += ((size_t)n * sizeof(P) + 255) / 256 * 256;
  };
  auto lay = [&] {
    at = 0;
    carve(&B.cn, 3, true);
    carve(&B.out, 16, true);
    for (RdFront& F : B.F) {
      carve(&F.v, fcap, true);
      carve(&F.s, fcap, true);
      carve(&F.e, fcap, true);
      carve(&F.tile, tiles, true);
      carve(&F.rank, fcap, true);
      carve(&F.brank, fcap, true);
      carve(&F.share, fcap, !staged);
      carve(&F.base, fcap, !staged);
      carve(&F.r0, fcap, !staged);
      carve(&F.p0, fcap, !staged);
      carve(&F.touched, std::min<int64_t>(g->n, e_max + fcap), det);
    }
    carve(&B.share, f_max, staged);
    carve(&B.base, f_max, staged);
    carve(&B.key, f_max, sel);
    carve(&B.pe, f_max, sel);
    carve(&B.ptile, tiles, sel);
    carve(&B.pv, f_max, sel && det);
    carve(&B.pr, f_max, sel && det);
    carve(&B.touched, std::min<int64_t>(g->n, e_max), wide);
    if (fresh_keys)
      for (int k = 0; k < 3; k++) carve(&fresh_keys[k], std::min<int64_t>(g->n, e_max + fcap), true);
    if (level_c) carve(level_c, levels, levels > 0);
  };
  lay();
  if (at > M.slab_bytes) {
    dfree(ctx, M.slab);
    M.slab = nullptr;
    M.slab_bytes = 0;
    const int st = take(&M.slab, at);
    if (st != LGC_OK) return *no_room ? LGC_OK : st;
    M.slab_bytes = at;
  }
  base = M.slab;
  lay();
  B.fcap = (int32_t)fcap;
  B.tiles = (int32_t)tiles;
  B.bucket = M.bucket;
  if (det || wide) {
    if (M.slots != slots) {
      dfree(ctx, M.per_slot);
      M.per_slot = nullptr;
      M.slots = 0;
      const size_t bytes = (4 + (wide ? sizeof(Fx) : 0)) * (size_t)slots;
      const int st = take(&M.per_slot, bytes);
      if (st != LGC_OK) return *no_room ? LGC_OK : st;
      M.slots = slots;
      LGC_CUDA_TRY(cudaMemsetAsync(M.per_slot, 0, bytes, s));
    }
    // the sums first: they need 16-byte alignment
    B.xacc = wide ? reinterpret_cast<Fx*>(M.per_slot) : nullptr;
    B.cnt = reinterpret_cast<int32_t*>(M.per_slot + (wide ? sizeof(Fx) * slots : 0));
  }
  LGC_CUDA_TRY(cudaMemsetAsync(B.cn, 0, 3 * sizeof(RdCnt), s));
  A.off = g->off;
  A.col = g->col;
  A.deg = g->deg;
  A.in_v = fv;
  A.in_s = fs;
  A.in_nf = nf;
  A.need_rank = rd_ranks(g) ? 1 : 0;
  A.gbits = 1;  // sums of at most max_deg terms: max_deg < 2^gbits
  while (A.gbits < 62 && (int64_t{1} << A.gbits) <= g->max_deg) A.gbits++;
  A.keep_room = fcap < g->n ? 1 : 0;
  A.x_min = det ? INT64_MAX : x_min;
  A.max_rounds = std::min<int64_t>(max_rounds, kRdRounds);
  A.e_max = e_max;
  A.f_max = f_max;
  A.key_limit = key_limit;
  A.hot = g->hot;
  return LGC_OK;
}

// Launches kern with args and reads the state it ended in.
int rd_run(lgc_ctx* ctx, lgc_graph* g, const void* kern, void** args, const RdBuf& B, bool det,
           RoundsOut* out) {
  cudaStream_t s = ctx->stream;
  const size_t smem = det ? (size_t)kRdSmemWords * 4 : 0;
  LGC_CUDA_TRY(
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  {
    ProfScope ps(ctx, det ? LGC_PROF_DET_EDGE : LGC_PROF_EDGEMAP, 0.0);
    // one block per SM: the rounds are small, and fewer blocks wait at each
    // grid barrier
    LGC_CUDA_TRY(cudaLaunchCooperativeKernel(kern, ctx->sms, kRdBlock, args, smem, s));
    LGC_COUNT_LAUNCH(ctx);
  }
  LGC_CUDA_TRY(cudaMemcpyAsync(ctx->h_scratch, B.out, 80, cudaMemcpyDeviceToHost, s));
  LGC_CUDA_TRY(cudaStreamSynchronize(s));
  const int64_t* o = ctx->h_scratch;
  if (o[0] != 0) return LGC_ETABLEFULL;
  if (o[5] < 1) return LGC_ECUDA;  // the caller checked that the first round is one to take
  const int cur = (int)o[1];
  out->v = B.F[cur].v;
  out->s = B.F[cur].s;
  out->nf = o[2];
  out->E = o[3];
  out->count = o[4];
  out->rounds = o[5];
  out->pushes = o[6];
  out->pushed = o[7];
  out->tab = (int)o[8];
  out->pcount = o[9];
  if (ctx->profile && !ctx->prof_pending.empty())
    ctx->prof_pending.back().bytes += 24.0 * (double)out->pushed + 88.0 * (double)out->pushes;
  // host-driven deterministic rounds take the frontier in ascending id
  if (det && out->nf > 1)
    LGC_TRY(radix_sort_u32_i32(ctx, (uint32_t*)out->v, out->s, (uint32_t*)B.F[cur ^ 1].v,
                               B.F[cur ^ 1].s, out->nf, bits_for(g->n)));
  return LGC_OK;
}

}  // namespace

int rounds_prnibble(lgc_ctx* ctx, lgc_graph* g, RoundsMem& M, const Table& T, const int32_t* fv,
                    const int32_t* fs, int64_t nf, int64_t E, int64_t count, double alpha,
                    double cs, double cn, double eps, int rule, bool det, double beta,
                    int64_t x_min, int64_t max_rounds, int64_t key_limit, RoundsOut* out) {
  (void)E;
  const bool sel = beta < 1.0;
  RdKernel kern = det ? (sel ? rounds_det_kernel<true> : rounds_det_kernel<false>)
                      : (sel ? rounds_kernel<true> : rounds_kernel<false>);
  RdLaunch L;
  bool no_room;
  LGC_TRY(rd_prepare(ctx, g, M, T.cap, fv, fs, nf, det, sel, !det || sel, x_min, max_rounds,
                     key_limit, nullptr, 0, nullptr, &L, &no_room));
  if (no_room) return LGC_OK;
  L.A.alpha = alpha;
  L.A.cs = cs;
  L.A.cn = cn;
  L.A.eps = eps;
  L.A.beta = beta;
  L.A.rule = rule;
  L.A.count = count;
  Table Tk = T;
  void* args[] = {&L.A, &L.B, &Tk};
  return rd_run(ctx, g, (const void*)kern, args, L.B, det, out);
}

int rounds_fresh(lgc_ctx* ctx, lgc_graph* g, RoundsMem& M, const RoundsFresh& q, const Table* T,
                 const Table* P, int64_t pcount, const int32_t* fv, const int32_t* fs, int64_t nf,
                 int64_t E, bool det, int64_t x_min, int64_t max_rounds, int64_t key_limit,
                 int64_t p_limit, RoundsOut* out) {
  (void)E;
  const bool hk = q.c != nullptr;
  RdLaunch L;
  RfArgs X{};
  RfTabs Q{};
  bool no_room;
  double* c = nullptr;
  LGC_TRY(rd_prepare(ctx, g, M, T[0].cap, fv, fs, nf, det, false, true, x_min, max_rounds,
                     key_limit, Q.keys, hk ? q.N + 1 : 0, &c, &L, &no_room));
  if (no_room) return LGC_OK;
  if (hk) {
    LGC_CUDA_TRY(cudaMemcpyAsync(c, q.c, sizeof(double) * (q.N + 1), cudaMemcpyHostToDevice,
                                 ctx->stream));
    X.t = q.t;
    X.c = c;
    X.N = q.N;
    X.j0 = q.j;
    X.pcount = pcount;
    X.p_limit = p_limit;
    Q.P = *P;
  }
  L.A.eps = q.eps;
  L.A.count = q.count;
  for (int k = 0; k < 4; k++) Q.T[k] = T[k];
  const void* kern = det ? (hk ? (const void*)rounds_fresh_kernel<true, 1>
                               : (const void*)rounds_fresh_kernel<true, 0>)
                         : (hk ? (const void*)rounds_fresh_kernel<false, 1>
                               : (const void*)rounds_fresh_kernel<false, 0>);
  void* args[] = {&L.A, &X, &L.B, &Q};
  return rd_run(ctx, g, kern, args, L.B, det, out);
}

}  // namespace lgc
