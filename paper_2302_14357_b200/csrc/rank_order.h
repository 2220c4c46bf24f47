// The order in which scored candidates are ranked: score descending, then place ascending.  It is total whatever the scores, so
// the ranks of n candidates are 0 .. n - 1, each taken once.  Plain C++ as well, so that it can be checked without a device.
#pragma once
#include <string.h>

#ifdef __CUDACC__
#define TW_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define TW_HOST_DEVICE inline
#endif

namespace tw {

// Order-preserving integer image of a score: a < b as doubles <=> order_key(a) < order_key(b) as unsigned
// integers (-0 counts as +0; scores are never NaN).  The ranking loops compare these instead of doubles.
TW_HOST_DEVICE unsigned long long order_key(double x) {
  x += 0.0;
  unsigned long long u;
  memcpy(&u, &x, sizeof u);
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

// Is a candidate (key, place) ahead of another?
TW_HOST_DEVICE bool ranks_before(unsigned long long key, unsigned long long place, unsigned long long other_key, unsigned long long other_place) {
  return key > other_key || (key == other_key && place < other_place);
}

// A row's list is in the order of its values; the approximate logarithm of two neighbours may come out the other way round (3 ulp
// each).  Each score is replaced by the smallest one up to it: the list's order is then the order of its scores, ties by place,
// and no score is further from its logarithm than one of them was.
TW_HOST_DEVICE void settle_row(double* score, int n) {
  for (int j = 1; j < n; ++j) if (score[j] > score[j - 1]) score[j] = score[j - 1];
}

}  // namespace tw
