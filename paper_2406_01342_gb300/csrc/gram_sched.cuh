// Tiles and K-shares of the tensor-core support contraction (gram_tc.cu): which
// rows, columns and stages of 16 visibilities each CTA takes. Host and device.
#pragma once

#include "pc_internal.cuh"

namespace pc {

constexpr int GB_M = 128;               // MMA M (rows of the A tile)
constexpr int GB_SUB = 16;              // stages per TMEM sub-slice (256 visibilities)

// One CTA's share: rows [a0, a0 + 128), columns [b0, b0 + n), `count` stages
// from `first`.
struct GbUnit {
  int a0, b0;
  int n;
  int first, count;
};

// Column chunks of a row tile whose first column is c0 (rows: columns in all):
// their number, and the width of all but the last (a multiple of 16).
__host__ __device__ __forceinline__ int gb_chunks(int rows, int c0, int* width) {
  const int cols = rows - c0, chunks = (cols + 255) / 256;
  *width = ((cols + chunks - 1) / chunks + 15) / 16 * 16;
  return chunks;
}
__host__ __device__ __forceinline__ int gb_width(int rows, int b0, int width) {
  const int left = (rows - b0 + 15) / 16 * 16;
  return left < width ? left : width;
}

// CTA `cta`: K-range cta / tiles of `stages` stages, tile cta % tiles in
// row-tile order, so the tiles of a range run next to each other.
__host__ __device__ __forceinline__ GbUnit gb_unit(int cta, int tiles, int stages, int n_stages, int rows) {
  const int z = cta / tiles;
  int t = cta - z * tiles;
  GbUnit u;
  u.a0 = 0;
  int w, c;
  while (t >= (c = gb_chunks(rows, u.a0, &w))) {
    t -= c;
    u.a0 += GB_M;
  }
  u.b0 = u.a0 + t * w;
  u.n = gb_width(rows, u.b0, w);
  u.first = z * stages;
  u.count = n_stages - u.first < stages ? n_stages - u.first : stages;
  return u;
}

// SM cycles of one stage: shared memory serves 128 bytes a cycle, to the six
// MMAs (the 4 KB of A and 32 n bytes of B that each reads) and from the copies
// (128 bytes a row). At n = 256 that is 960 against the tensor pipe's 768, at
// n = 128 640 against 384.
inline int64_t gb_stage_cycles(int n, bool diag) {
  return 192 + 3 * n / 2 + (diag ? std::max(n, GB_M) : n + GB_M);
}

// A CTA's start and end (pipeline fill, flush of 128 x n reductions), in
// stages of 256 columns (0.5 us each): about 6 us.
constexpr int GB_OVERHEAD = 12;

// Stages per K-slice: FP32 sums run over a slice, float64 over the slices, so
// the slice length is part of the result's rounding. It is the one that fills
// whole waves with the slices of 128 x 256 tiles. It stays what it is whatever
// the CTAs below take: the restricted LASSO of neighbouring pixels passes a
// change of G's last bits on a hundredfold (5e-7 in G moved weights of 512 x
// 512 solves by up to 5e-5, and the iterations a stop takes).
inline int gb_slice(int rows, int nA, int n_stages, int n_sm) {
  const int w = rows > 128 ? 256 : (rows > 64 ? 128 : 64);
  int64_t tiles = 0;
  for (int a0 = 0; a0 < nA; a0 += GB_M)
    for (int b0 = 0; b0 < rows; b0 += w) tiles += b0 + w > a0;
  int best_z = 1;
  int64_t best = INT64_MAX;
  for (int z = 1; z <= std::max(1, n_stages / GB_SUB); ++z) {
    const int64_t c = (int64_t)ceil_div(tiles * z, n_sm) * ceil_div(n_stages, z);
    if (c < best) {
      best = c;
      best_z = z;
    }
  }
  return ceil_div(n_stages, best_z);
}

struct GbPlan {
  int tiles = 0;    // row tiles x column chunks
  int slice = 0;    // stages per K-slice
  int stages = 0;   // stages per CTA: whole slices
  int ctas = 0;
  int widest = 0;   // columns of the widest tile
};

// The K-range of a CTA: the number of slices with the least time on the busiest
// SM, in whole waves of the widest tile (narrower tiles to fill the last wave,
// 224 or 192 columns, measured between 1.5 % faster and 11 % slower and are left
// out). Ranges stay contiguous in K: CTAs that
// took every m-th stage of one common sweep instead, m by tile width, measured
// 1.4 times slower (873 atoms, 200k visibilities: 1.09 against 0.74 ms).
inline GbPlan gb_schedule(int rows, int nA, int n_stages, int n_sm) {
  GbPlan p;
  int64_t wide = 0;
  for (int a0 = 0; a0 < nA; a0 += GB_M) {
    int w;
    const int chunks = gb_chunks(rows, a0, &w);
    p.tiles += chunks;
    const int n0 = gb_width(rows, a0, w);
    p.widest = std::max(p.widest, n0);
    wide = std::max(wide, chunks > 1 ? gb_stage_cycles(w, false) : gb_stage_cycles(n0, true));
  }
  p.slice = gb_slice(rows, nA, n_stages, n_sm);
  const int slices = ceil_div(n_stages, p.slice);
  int64_t best = INT64_MAX;
  for (int per = slices; per >= 1; --per) {
    const int64_t waves = ceil_div((int64_t)p.tiles * ceil_div(slices, per), n_sm);
    const int64_t c = waves * wide * ((int64_t)per * p.slice + GB_OVERHEAD);
    if (c < best) {
      best = c;
      p.stages = per * p.slice;
    }
  }
  p.ctas = p.tiles * ceil_div(n_stages, p.stages);
  return p;
}

}  // namespace pc
