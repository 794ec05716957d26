// Consecutive small PR-Nibble rounds in one cooperative launch (rounds.cu).
#pragma once

#include "common.cuh"

namespace lgc {

// The device memory of the rounds kernels, kept by one run's push state: one
// slab for the frontier buffers and lists, the per-slot counters of
// deterministic rounds or counters and sums of wide atomic rounds (zero
// between launches; a run keeps one mode), and the deterministic rounds'
// buckets (4 bytes per adjacency entry; no_det: there was no room for them).
struct RoundsMem {
  char* slab = nullptr;
  size_t slab_bytes = 0;
  char* per_slot = nullptr;
  int64_t slots = 0;
  int32_t* bucket = nullptr;
  bool no_det = false;
  void release(lgc_ctx* ctx) {
    dfree(ctx, slab);
    dfree(ctx, per_slot);
    dfree(ctx, bucket);
    *this = RoundsMem();
  }
};

// The state the rounds ran to.  v, s: the frontier reached (device pointers
// into the slab, valid until its next use; ascending by vertex in
// deterministic mode), nf entries with degree sum E.
struct RoundsOut {
  int32_t *v = nullptr, *s = nullptr;
  int64_t nf = 0, E = 0, count = 0, rounds = 0, pushes = 0, pushed = 0;
};

// Whether the rounds kernel takes a frontier of nf vertices and E edges
// (sets that stay within key_limit keys are the caller's concern).
bool rounds_take(const lgc_ctx* ctx, const lgc_graph* g, const RoundsMem& M, int64_t nf, int64_t E,
                 bool det, bool beta);

// Runs PR-Nibble rounds from the frontier (fv, fs)[0, nf) with the sets in T
// (count keys) until the frontier is empty, max_rounds have run or the next
// round is not one for the device; runs at least one round when rounds_take
// holds, count + E is within key_limit and max_rounds > 0.  Atomic rounds of
// x_min edges or more sum as pull rounds do.  rounds 0 in *out: there was no
// room (M.no_det is set), nothing has changed.
int rounds_prnibble(lgc_ctx* ctx, lgc_graph* g, RoundsMem& M, const Table& T, const int32_t* fv,
                    const int32_t* fs, int64_t nf, int64_t E, int64_t count, double alpha,
                    double cs, double cn, double eps, int rule, bool det, double beta,
                    int64_t x_min, int64_t max_rounds, int64_t key_limit, RoundsOut* out);

}  // namespace lgc
