// Host check of the skewed tiles' 32-bit row arithmetic (fx/skew.cuh, compiled
// by tests/test_skew_extent.py and run on the CPU): for every extent that
// skew_extent accepts, the last tile's first row, its end and the rows of its
// last vectors fit in 32 bits, for each tile height, vector width and shift.
#include <climits>
#include <cstdio>

#include "fx/batch.cuh"

int main() {
  long bad = 0, checked = 0;
  const int64_t top = int64_t(1) << 31;
  bad += fx::skew_extent(top - 1, 1) + fx::skew_extent(1, top - 1) + fx::skew_extent(top, 1);
  bad += !fx::skew_extent(int64_t(1) << 30, 1) + !fx::skew_extent(1, int64_t(1) << 30);
  for (int64_t R = top - 1; R > top - 512; --R) {
    if (!fx::skew_extent(R, 1)) continue;
    for (int TR : {32, 64})
      for (int V : {2, 4, 8})
        for (int shift = 0; shift < V; ++shift) {
          const int64_t tiles = (R + shift + TR - 1) / TR, r0 = (tiles - 1) * TR;
          ++checked;
          bad += r0 + TR > INT_MAX || r0 + TR + 2 * V > INT_MAX;  // skew_tile's test, a row and its vector
        }
  }
  printf("checked %ld bad %ld\n", checked, bad);
  return 0;
}
