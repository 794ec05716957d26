// Consecutive small rounds in one cooperative launch (rounds.cu).
#pragma once

#include "common.cuh"

namespace lgc {

// The device memory of the rounds kernels, kept by one run's push state: one
// slab for the frontier buffers and lists, the per-slot counters of
// deterministic rounds or counters and sums of wide atomic rounds (zero
// between launches; a run keeps one mode), and the deterministic rounds'
// buckets (4 bytes per adjacency entry).  no_room: there was no device memory
// for one of them; the run's rounds stay on the host.
struct RoundsMem {
  char* slab = nullptr;
  size_t slab_bytes = 0;
  char* per_slot = nullptr;
  int64_t slots = 0;
  int32_t* bucket = nullptr;
  bool no_room = false;
  void release(lgc_ctx* ctx) {
    dfree(ctx, slab);
    dfree(ctx, per_slot);
    dfree(ctx, bucket);
    *this = RoundsMem();
  }
  void give_up(lgc_ctx* ctx) {
    release(ctx);
    no_room = true;
  }
};

// The state the rounds ran to.  v, s: the frontier reached (device pointers
// into the slab, valid until its next use; ascending by vertex in
// deterministic mode), nf entries with degree sum E.
struct RoundsOut {
  int32_t *v = nullptr, *s = nullptr;
  int64_t nf = 0, E = 0, count = 0, rounds = 0, pushes = 0, pushed = 0;
  int tab = 3;         // fresh sets: which table holds the set reached (3: the first)
  int64_t pcount = 0;  // HK-PR: keys of p
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
// room (M.no_room is set), nothing has changed.
int rounds_prnibble(lgc_ctx* ctx, lgc_graph* g, RoundsMem& M, const Table& T, const int32_t* fv,
                    const int32_t* fs, int64_t nf, int64_t E, int64_t count, double alpha,
                    double cs, double cn, double eps, int rule, bool det, double beta,
                    int64_t x_min, int64_t max_rounds, int64_t key_limit, RoundsOut* out);

// Rounds that fill a fresh set from the frontier: Nibble (c null; threshold
// eps, 0: every inserted vertex goes on) or HK-PR from level j of N (t, and
// the levels' threshold factors c[0..N]).
struct RoundsFresh {
  double eps = 0.0, t = 0.0;
  const double* c = nullptr;
  int N = 0, j = 0;
  int64_t count = 0;  // keys of the first set
};

// Runs such rounds: the first reads the set T[3], the others T[0..2] in turn
// (cleared, of one form; key_limit keys each).  HK-PR adds into P (pcount
// keys, at most p_limit) and stops before its last level.  Nibble stops with
// an empty frontier at the round that made it, T[tab] being the vector before
// that round, as the method returns it.  rounds 0 in *out: as above.
int rounds_fresh(lgc_ctx* ctx, lgc_graph* g, RoundsMem& M, const RoundsFresh& q, const Table* T,
                 const Table* P, int64_t pcount, const int32_t* fv, const int32_t* fs, int64_t nf,
                 int64_t E, bool det, int64_t x_min, int64_t max_rounds, int64_t key_limit,
                 int64_t p_limit, RoundsOut* out);

}  // namespace lgc
