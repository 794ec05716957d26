// FP64 with less of it.  GB300 issues a warp's FP64 instruction every 20
// cycles or so per SM (498 G adds/s on the device, a few percent of the
// integer rate), so kernels that do little else than a compare against a
// threshold c * d(v) or a division per vertex are bound by that pipe: the
// dense filter over 4.2M vertices spent 40 us at 79% of it (now 21), the HK-PR
// vertexMap of 2.3M 64 us at 83% (now 47), the sweep's keys 64 us.  The same
// results with integer and FP32 instructions, or with fewer FP64 ones.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define LGC_LITE __host__ __device__ __forceinline__
#else
#define LGC_LITE inline
#include <math.h>
#include <string.h>
#endif

namespace lgc {

LGC_LITE uint32_t lite_hi(double x) {
#if defined(__CUDA_ARCH__)
  return (uint32_t)__double2hiint(x);
#else
  uint64_t b;
  __builtin_memcpy(&b, &x, 8);
  return (uint32_t)(b >> 32);
#endif
}
LGC_LITE uint32_t lite_bits(float x) {
#if defined(__CUDA_ARCH__)
  return __float_as_uint(x);
#else
  uint32_t b;
  __builtin_memcpy(&b, &x, 4);
  return b;
#endif
}

// A threshold c * d(v): cf is c in single precision, 0 where c leaves the
// range in which the products of lite_reaches are normal floats.
struct LiteThr {
  double c;
  float cf;
};
LGC_LITE LiteThr lite_thr(double c) {
  return {c, c > 1e-30 && c < 1e20 ? (float)c : 0.0f};
}

// x >= c * (double)d (one rounding, as that expression), for x >= 0 and
// 1 <= d < 2^31.  t = cf * (float)d is within 2^-22 of c * d, so the high
// words h(t) and h(c d) (20 mantissa bits: a unit is at least 2^-21 of the
// value) differ by at most one.  h(x) >= h(t) + 2 then puts a multiple of the
// unit, a double, between c d and x, and x is at least the rounded product;
// h(x) <= h(t) - 2 puts one above x and at or below c d.  In between the
// expression itself decides.
LGC_LITE bool lite_reaches(double x, LiteThr T, int32_t d) {
  if (T.cf != 0.0f) {
    const float t = T.cf * (float)d;
    const uint32_t ht = (lite_bits(t) >> 3) + ((1023u - 127u) << 20);
    const int32_t diff = (int32_t)((lite_hi(x) & 0x7FFFFFFFu) - ht);
    if (diff >= 2) return true;
    if (diff <= -2) return false;
  }
  return x >= T.c * (double)d;
}

// 1 / b to twice the precision: h = RN(1/b), l the rest.
struct __attribute__((aligned(16))) Recip {
  double h, l;
};
LGC_LITE Recip recip_of(double b) {
  const double h = 1.0 / b;
#if defined(__CUDA_ARCH__)
  return {h, __fma_rn(-b, h, 1.0) * h};
#else
  return {h, fma(-b, h, 1.0) * h};
#endif
}

// RN(a / b) from y = recip_of(b), for a >= 0 and an integer 1 <= b <= 2^48:
// a y in double-double (one product, its exact error, one more term, one
// sum) in place of the division's iteration.  The double-double is within
// 2^-104 of a/b.  a/b lies at least 2^-54 / b of it away from any midpoint of
// two doubles unless it is one, and it is none: 2 A = M b 2^k with M odd and
// of 54 bits needs A of more than 53 bits for every b but a power of two,
// for which a/b is a double.  So the rounded sum is the rounded quotient.
// Where a's exponent could make a term underflow or overflow the division
// itself is used.
LGC_LITE double div_by(double a, Recip y, double b) {
  const uint32_t be = lite_hi(a) >> 20;
  if (be - 160u < 1700u) {
    const double p = a * y.h;
#if defined(__CUDA_ARCH__)
    return p + __fma_rn(a, y.l, __fma_rn(a, y.h, -p));
#else
    return p + fma(a, y.l, fma(a, y.h, -p));
#endif
  }
  return a / b;
}

// Degrees with an entry in a graph's table of reciprocals.
constexpr int32_t kRecipMax = 1 << 20;

}  // namespace lgc
