// Host-side check of the rows that the LASSO cluster's CTAs take (apgd_rows.cuh):
// for every size above the one-CTA kernel's and every cluster size, each CTA has
// rows, they start at a multiple of 4, number at most cluster_rows(), and follow one
// another from the first row to the last.
// Prints "ok" and exits 0, or the first failure and exits 1.
#include "apgd_rows.cuh"

#include <cstdio>

int main() {
  for (int n = 225; n <= 7200; ++n)
    for (int cs = 1; cs <= 16; cs *= 2) {
      int next = 0;
      for (int rank = 0; rank < cs; ++rank) {
        const pc::RowSlice s = pc::cluster_slice(n, cs, rank);
        if (s.r0 != next || s.r0 % 4 || s.nr < 1 || s.nr > pc::cluster_rows(n, cs)) {
          std::printf("n %d, CTA %d of %d: rows %d + %d, expected from %d\n", n, rank, cs, s.r0, s.nr, next);
          return 1;
        }
        next = s.r0 + s.nr;
      }
      if (next != n) {
        std::printf("n %d on %d CTAs: rows end at %d\n", n, cs, next);
        return 1;
      }
    }
  std::printf("ok\n");
  return 0;
}
