// Host build of fp64lite.cuh for tests/test_fp64lite_host.py.
#include <stdint.h>

#include "../paper_1604_07515_gb300/csrc/fp64lite.cuh"

extern "C" {
// The number of entries where the short form differs from the expression.
int64_t reaches_bad(int64_t n, const double* x, const double* c, const int32_t* d) {
  int64_t bad = 0;
  for (int64_t i = 0; i < n; i++)
    bad += lgc::lite_reaches(x[i], lgc::lite_thr(c[i]), d[i]) != (x[i] >= c[i] * (double)d[i]);
  return bad;
}
int64_t div_bad(int64_t n, const double* a, const double* b) {
  int64_t bad = 0;
  for (int64_t i = 0; i < n; i++)
    bad += lgc::div_by(a[i], lgc::recip_of(b[i]), b[i]) != a[i] / b[i];
  return bad;
}
}
