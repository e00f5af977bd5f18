// Rows of G of each CTA of the full-vector LASSO kernel's cluster (apgd.cu). Host
// and device.
#pragma once

namespace pc {

struct RowSlice {
  int r0, nr;   // rows [r0, r0 + nr)
};

// Most rows of a CTA: whole groups of four.
__host__ __device__ __forceinline__ int cluster_rows(int n, int cs) { return ((n + 3) / 4 + cs - 1) / cs * 4; }

// The groups of four dealt out evenly, so that every CTA of a cluster of at most (n +
// 3) / 4 has rows. Equal slices of cluster_rows() would leave the last CTAs none
// (257 atoms on 16 CTAs: 20 rows each, three without), and the exchange needs a
// contribution of every CTA: it is what keeps the others from sending product i + 2
// into a buffer that a CTA still reads product i from.
__host__ __device__ __forceinline__ RowSlice cluster_slice(int n, int cs, int rank) {
  const int groups = (n + 3) / 4;
  const int r0 = 4 * (int)((long long)groups * rank / cs), r1 = 4 * (int)((long long)groups * (rank + 1) / cs);
  return {r0, (r1 < n ? r1 : n) - r0};
}

}  // namespace pc
