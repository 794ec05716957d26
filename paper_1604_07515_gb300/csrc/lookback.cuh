// Decoupled look-back (Merrill and Garland's single-pass prefix scan): the
// status words the one-launch scans and sorts publish per tile and the
// warp-wide look-back over them; and the ordered compaction of a vertex
// bitmap (or of one computed word by word), which does without a look-back.
//
// A status word: epoch (24 bits) | state (2 bits: aggregate, inclusive
// prefix) | value (38 bits).  Every launch (every radix pass) has its own
// epoch, so the status array is cleared only when it is (re)allocated or the
// epochs wrap; a word of another epoch is "not yet published".  A look-back
// wait that exceeds kLbSpinLimit polls (it cannot, as every earlier tile's
// block is running) records the failure in *err and counts the tile as
// empty.
#pragma once

#include "common.cuh"

namespace lgc {

constexpr uint64_t kLbValue = (1ull << 38) - 1;
constexpr uint64_t kLbAggregate = 1ull << 38;
constexpr uint64_t kLbInclusive = 2ull << 38;
constexpr int kLbSpinLimit = 1 << 22;

__device__ inline uint64_t lb_word(uint32_t epoch, uint64_t state, uint64_t count) {
  return ((uint64_t)epoch << 40) | state | count;
}

// A value of a single-value status word: 38-bit two's complement.
__device__ inline int64_t lb_value(uint64_t w) { return (int64_t)(w << 26) >> 26; }

// Look-back by one whole warp for tiles with one status word each: the sum
// of the values of tiles [0, t), lane l reading tile j - l of a 32-tile
// window, the walk ending at the nearest inclusive word.  The warp waits
// until every word of the window is published (bounded: past kLbSpinLimit
// polls *err records it and unpublished words count as empty inclusive
// ones).  Every lane of the warp calls it and gets the sum.
__device__ inline int64_t lookback_warp(const unsigned long long* status, int64_t t,
                                        uint32_t epoch, int* err) {
  const int lane = threadIdx.x & 31;
  int64_t excl = 0;
  for (int64_t j = t - 1; j >= 0; j -= 32) {  // uniform in the warp
    const int64_t tj = j - lane;
    const volatile unsigned long long* pj = status + (tj >= 0 ? tj : 0);
    uint64_t w = tj >= 0 ? *pj : lb_word(epoch, kLbInclusive, 0);
    for (int spins = 0;; spins++) {
      const bool ready = (uint32_t)(w >> 40) == epoch;
      if (__all_sync(0xffffffffu, ready)) break;
      if (spins > kLbSpinLimit) {  // the same count in every lane
        if (lane == 0) atomicOr(err, 1);
        if (!ready) w = lb_word(epoch, kLbInclusive, 0);
        break;
      }
      if (spins > 16) __nanosleep(64);
      if (!ready) w = *pj;
    }
    const unsigned incl = __ballot_sync(0xffffffffu, (w & kLbInclusive) != 0);
    const int last = incl ? __ffs(incl) - 1 : 31;  // lanes 0..last count
    int64_t v = lane <= last ? lb_value(w) : 0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    excl += v;
    if (incl) break;
  }
  return excl;
}

// ---------------------------------------------------------------------------
// Ordered compaction of a vertex bitmap in two launches (three for graphs of
// more than 2^24 vertices).  The bitmap's words
// come from a functor called by whole warps (word(w, in): lane l asks for
// word w = the warp's first + l, `in` saying whether it has one), so that a
// filter can compute them on the fly, 32 vertices of a word at a time with
// one lane each.  words_count_kernel keeps the words and counts the set bits
// of every tile of kCmpTileWords words; words_write_kernel adds up the counts
// of the tiles before its own (up to 2^22 vertices 8 loads a thread) and hands
// every set bit's vertex v to out.put(position, v), lane l with bit l
// of one word after another, so a warp's positions are consecutive.  put
// returns a weight, and out.finish(entries so far, is this the last tile,
// weight of the block's vertices) is called by one thread per tile.
//
// 4.2M vertices, 2.4M of them kept: 3 + 20 us (one launch with a decoupled
// look-back 27 us); the dense filter over them 21 + 12 us (30-37 us, with the
// lanes walking their own words' bits and FP64 compares, which alone bound it
// at 40 us); a look-back by the whole block instead of one warp 45-50 us (its
// polls crowd out the words it waits for).
// ---------------------------------------------------------------------------
constexpr int kCmpWarpWords = 8;  // words a warp writes: one batch of loads each
constexpr int64_t kCmpTileWords = kCmpWarpWords * (kBlock / 32);
// More tiles than kCmpPlain have their counts added up in groups of kCmpGroup
// first: adding those of all tiles before one's own is quadratic, nothing at
// 2^22 vertices but most of the pass from 2^26 on.  Both launches together, a
// 16th and half of the words not empty: 2^22 vertices 15 and 17 us (19 and 21
// with groups), 2^24 37 and 44 (37 and 44), 2^25 78 and 91 (66 and 78), 2^26
// 185 and 199 (119 and 138), 2^28 1565 and 1669 (443 and 543).
constexpr int kCmpGroup = 1024;
constexpr int64_t kCmpPlain = 8192;

template <class WordFn>
__global__ void __launch_bounds__(kBlock)
    words_count_kernel(WordFn word, int64_t words, uint32_t* __restrict__ kept,
                       int32_t* __restrict__ cnt) {
  __shared__ int s_tot[kBlock / 32], s_new[kBlock / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t w = (int64_t)blockIdx.x * kCmpTileWords + warp * kCmpWarpWords + lane;
  const bool in = lane < kCmpWarpWords && w < words;
  int fresh = 0;  // keys the functor found and marked
  const uint32_t q = word(w, in, &fresh);
  if (kept && in) kept[w] = q;
  const int c = __reduce_add_sync(0xffffffffu, __popc(q));
  fresh = __reduce_add_sync(0xffffffffu, fresh);
  if (lane == 0) {
    s_tot[warp] = c;
    s_new[warp] = fresh;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0, f = 0;
    for (int k = 0; k < kBlock / 32; k++) {
      t += s_tot[k];
      f += s_new[k];
    }
    cnt[blockIdx.x] = t;
    if (f) word.marked(f);
  }
}

template <class Out>
__global__ void __launch_bounds__(kBlock)
    words_write_kernel(const uint32_t* __restrict__ kept, int64_t words,
                       const int32_t* __restrict__ cnt, const int64_t* __restrict__ grp, Out out) {
  __shared__ int64_t s_pre[kBlock / 32];
  __shared__ int s_wtot[kBlock / 32];
  __shared__ int64_t s_sum[kBlock / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t tile = blockIdx.x;
  const int64_t wbase = tile * kCmpTileWords + warp * kCmpWarpWords;
  const uint32_t q = lane < kCmpWarpWords && wbase + lane < words ? kept[wbase + lane] : 0u;
  int64_t p = 0;
  const int64_t whole = grp ? tile / kCmpGroup : 0;  // groups before the tile's own
  for (int64_t i = threadIdx.x; i < whole; i += kBlock) p += grp[i];
  for (int64_t i = whole * kCmpGroup + threadIdx.x; i < tile; i += kBlock) p += cnt[i];
  for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
  const int c = __popc(q);
  int pre = c;  // set bits of the warp's words before this lane's
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, pre, o);
    if (lane >= o) pre += y;
  }
  if (lane == 31) s_wtot[warp] = pre;
  if (lane == 0) s_pre[warp] = p;
  pre -= c;
  __syncthreads();
  int64_t at = 0, tot = 0;
  for (int w = 0; w < kBlock / 32; w++) {
    at += s_pre[w];
    tot += s_wtot[w];
  }
  tot += at;  // entries through this tile
  for (int w = 0; w < warp; w++) at += s_wtot[w];
  const uint32_t below = (1u << lane) - 1u;
  int64_t sum = 0;
  if (__any_sync(0xffffffffu, q != 0u)) {
    int64_t x[kCmpWarpWords];
#pragma unroll
    for (int j = 0; j < kCmpWarpWords; j++) {
      const uint32_t qj = __shfl_sync(0xffffffffu, q, j);
      const int pj = __shfl_sync(0xffffffffu, pre, j);
      x[j] = (qj >> lane) & 1u ? out.put(at + pj + __popc(qj & below), (wbase + j) * 32 + lane)
                               : 0;
    }
#pragma unroll
    for (int j = 0; j < kCmpWarpWords; j++) sum += x[j];
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) s_sum[warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t t = 0;
    for (int w = 0; w < kBlock / 32; w++) t += s_sum[w];
    out.finish(tot, tile == gridDim.x - 1, t);
  }
}

// The bits of word w of a bitmap whose vertices v (< n) pass keep(v, x), by a
// whole warp: the words of its first kCmpWarpWords lanes, the lanes taking a
// word's vertices side by side.  x = load(v); all words' loads in flight.
template <class Load, class Keep>
__device__ inline uint32_t filter_words(uint32_t m, int64_t w, int64_t n, Load&& load,
                                        Keep&& keep) {
  const int lane = threadIdx.x & 31;
  const int64_t wb = w - lane;
  uint32_t q = 0;
  if (!__any_sync(0xffffffffu, m != 0u)) return 0;
  double x[kCmpWarpWords];
  bool p[kCmpWarpWords];
#pragma unroll
  for (int j = 0; j < kCmpWarpWords; j++) {
    const int64_t v = (wb + j) * 32 + lane;
    p[j] = ((__shfl_sync(0xffffffffu, m, j) >> lane) & 1u) && v < n;
    x[j] = p[j] ? load(v) : 0.0;
  }
#pragma unroll
  for (int j = 0; j < kCmpWarpWords; j++) p[j] = p[j] && keep((wb + j) * 32 + lane, x[j]);
#pragma unroll
  for (int j = 0; j < kCmpWarpWords; j++) {
    const uint32_t b = __ballot_sync(0xffffffffu, p[j]);
    if (lane == j) q = b;
  }
  return q;
}

// Compaction into a frontier: vertex ids (twice: dense slots are vertices),
// their number and the sum of their degrees.
struct FrontierOut {
  const int32_t* deg;
  int32_t *v, *s;
  int32_t cap;
  Counters* C;
  __device__ int64_t put(int64_t at, int64_t u) const {
    if (at < cap) {
      v[at] = (int32_t)u;
      s[at] = (int32_t)u;
    } else {
      atomicOr(&C->err, kErrFrontierOverflow);
    }
    return deg ? deg[u] : 0;
  }
  __device__ void finish(int64_t n, bool last, int64_t weight) const {
    if (last) C->next_size = (int32_t)n;
    if (weight) atomicAdd((unsigned long long*)&C->next_edges, (unsigned long long)weight);
  }
};

// The two launches on the context's scratch; bits: the words themselves where
// word only reads them (nothing is kept then), else nullptr.
int cmp_reserve(lgc_ctx* ctx, int64_t words, uint32_t** kept, int32_t** cnt, int64_t** grp);
// grp[b] = the sum of cnt[b * kCmpGroup ...] (kCmpGroup of them, or what is left).
int tile_groups(lgc_ctx* ctx, const int32_t* cnt, int64_t ntiles, int64_t* grp);

template <class WordFn, class Out>
int words_compact(lgc_ctx* ctx, const WordFn& word, const uint32_t* bits, int64_t words,
                  const Out& out) {
  if (words <= 0) return LGC_OK;
  const unsigned ntiles = (unsigned)((words + kCmpTileWords - 1) / kCmpTileWords);
  uint32_t* kept;
  int32_t* cnt;
  int64_t* grp;
  LGC_TRY(cmp_reserve(ctx, words, &kept, &cnt, &grp));
  words_count_kernel<WordFn><<<ntiles, kBlock, 0, ctx->stream>>>(word, words,
                                                                 bits ? nullptr : kept, cnt);
  LGC_COUNT_LAUNCH(ctx);
  const bool groups = ntiles > kCmpPlain;
  if (groups) LGC_TRY(tile_groups(ctx, cnt, ntiles, grp));
  words_write_kernel<Out><<<ntiles, kBlock, 0, ctx->stream>>>(bits ? bits : kept, words, cnt,
                                                              groups ? grp : nullptr, out);
  LGC_COUNT_LAUNCH(ctx);
  return cudaGetLastError() == cudaSuccess ? LGC_OK : LGC_ECUDA;
}

}  // namespace lgc
