// Host build of fx128.cuh's windowed sums for tests/test_fxwindow_host.py.
#include <stdint.h>

#define __align__(n) __attribute__((aligned(n)))
#include "../paper_1604_07515_gb300/csrc/fx128.cuh"

using namespace lgc;

extern "C" {
int win_windows(int be_min, int be_max, int g) {
  return fx_windows(be_min, be_max, fx_scale(be_min, be_max, g));
}
// The sum of n shares in w windows and term by term; 0 if they are equal.
int win_differs(int w, int64_t n, const double* x, int be_min, int be_max, int g) {
  const int L = fx_scale(be_min, be_max, g);
  Fx t = {0, 0};
  FxWindow<1> a;
  FxWindow<2> b;
  for (int64_t i = 0; i < n; i++) {
    fx_add(t, fx_from_bits(fx_bits(x[i]), L));
    if (w == 1) a.add(fx_bits(x[i]), (uint32_t)be_min);
    else b.add(fx_bits(x[i]), (uint32_t)be_min);
  }
  const Fx s = w == 1 ? a.total() : b.total();
  return s.lo != t.lo || s.hi != t.hi;
}
}
