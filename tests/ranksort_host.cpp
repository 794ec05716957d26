// Host build of ranksort.cuh for tests/test_ranksort_host.py.
#include "../paper_1604_07515_gb300/csrc/ranksort.cuh"

extern "C" int rank_takes(int64_t n, int digits) { return lgc::rank_sort_takes(n, digits); }
