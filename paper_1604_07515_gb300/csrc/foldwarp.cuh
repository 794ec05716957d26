// The warp-wide ordered fold shared by the deterministic gathers, the folds of
// long destination runs and the device-driven deterministic rounds.
#pragma once

#include "fx128.cuh"

namespace lgc {

// ---------------------------------------------------------------------------
// The ordered fold acc <- RN(acc + s_k) of 256 shares by a warp, without a
// chain of dependent FP64 adds (the segment-parallel fold of long lists
// refolds a segment with it where its composed step does not apply).
//
// While acc stays in one binade it is A * u with the integer A below 2^53,
// and each share is an integer step A -> A + g[A & 1] (fold_step in
// fx128.cuh); steps compose, so a warp scan of the compositions gives every
// partial fold.  The first position whose value reaches 2^53 leaves the
// binade: that one add is done in FP64 (the rounding of the next binade
// applies), and the scan restarts after it with the new binade.  Every
// result equals the sequential fold's bit for bit.
// ---------------------------------------------------------------------------
// Folds the 32 * NL shares v (lane l holds positions NL l .. NL l + NL - 1, in
// list order) into acc, lane-uniformly.
template <int NL = 8>
__device__ inline double fold_batch(double acc, const double (&v)[NL], int lane) {
  int start = 0;
  while (start < 32 * NL) {
    const int bu = fold_binade(acc);
    const int64_t A0 = fold_int(acc);
    // the lane's steps from an even and from an odd value
    int64_t d[NL];
    uint32_t tie = 0;
    int64_t x0 = 0, x1 = 1;
#pragma unroll
    for (int j = 0; j < NL; j++) {
      FoldNear f = fold_near(v[j], bu);
      if (NL * lane + j < start) f = {0, false};
      d[j] = f.d;
      tie |= (uint32_t)f.tie << j;
      x0 = fold_take(f, x0);
      x1 = fold_take(f, x1);
    }
    // exclusive scan over lanes.  A step depends on the value's parity only at
    // a tie: without one among them the compositions are plain sums
    int64_t A;
    if (!__any_sync(0xffffffffu, tie != 0)) {
      int64_t P = x0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t q = __shfl_up_sync(0xffffffffu, P, o);
        if (lane >= o) P += q;
      }
      A = A0 + (P - x0);
    } else {
      FoldStep P = {x0, x1 - 1}, E;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        FoldStep q;
        q.g0 = __shfl_up_sync(0xffffffffu, P.g0, o);
        q.g1 = __shfl_up_sync(0xffffffffu, P.g1, o);
        if (lane >= o) P = fold_compose(q, P);
      }
      E.g0 = __shfl_up_sync(0xffffffffu, P.g0, 1);
      E.g1 = __shfl_up_sync(0xffffffffu, P.g1, 1);
      if (lane == 0) E = {0, 0};
      A = fold_apply(E, A0);
    }
    int cj = -1;
    int64_t before = 0;
#pragma unroll
    for (int j = 0; j < NL; j++) {
      const int64_t nx = fold_take({d[j], (tie >> j & 1u) != 0}, A);
      if (cj < 0 && nx >= kFoldTop) {
        cj = j;
        before = A;
      }
      A = nx;
    }
    const unsigned crossed = __ballot_sync(0xffffffffu, cj >= 0);
    if (!crossed) {
      const int64_t Aend = __shfl_sync(0xffffffffu, A, 31);
      return fold_double(Aend, bu);
    }
    const int lc = __ffs(crossed) - 1;
    double nacc = 0.0;
    if (lane == lc) {
      double sj = 0.0;
#pragma unroll
      for (int j = 0; j < NL; j++)
        if (j == cj) sj = v[j];
      nacc = fold_double(before, bu) + sj;  // the add that leaves the binade
    }
    acc = __shfl_sync(0xffffffffu, nacc, lc);
    start = NL * lc + __shfl_sync(0xffffffffu, cj, lc) + 1;
  }
  return acc;
}

}  // namespace lgc
