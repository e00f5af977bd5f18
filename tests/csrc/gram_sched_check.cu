// Host-side check of the support contraction's schedule (gram_sched.cuh): for
// many (rows, new atoms, stages, SMs) every entry the caller reads (column >=
// row, or any column beyond the new atoms) is covered by exactly one tile, the
// CTAs of a tile take every stage exactly once, tile widths are valid MMA
// shapes, and no tile reads a row beyond the padded phase buffer.
// Prints "ok" and exits 0, or the first failure and exits 1.
#include "gram_sched.cuh"

#include <cstdio>
#include <map>
#include <random>
#include <vector>

using namespace pc;

int main() {
  std::mt19937 rng(7);
  for (int trial = 0; trial < 1500; ++trial) {
    const int nA = trial < 40 ? 1 + trial * 13 : 1 + (int)(rng() % (trial % 3 ? 1200 : 5000));
    const int rows = nA + (int)(rng() % 3 ? rng() % 2 : rng() % 2000);
    const int n_stages = trial % 5 == 0 ? 1 + (int)(rng() % 20) : 1 + (int)(rng() % 20000);
    const int n_sm = trial % 2 ? 152 : 148;
    const GbPlan p = gb_schedule(rows, nA, n_stages, n_sm);
    const int rows_pad = std::max(ceil_div(rows, 16) * 16, ceil_div(nA, GB_M) * GB_M);
    std::map<std::pair<int, int>, std::vector<GbUnit>> by_tile;
    for (int c = 0; c < p.ctas; ++c) {
      const GbUnit u = gb_unit(c, p.tiles, p.stages, n_stages, rows);
      if (p.stages % p.slice || u.n % 16 || u.n < 16 || u.n > 256 || u.n > p.widest || u.a0 % GB_M || u.b0 % 16 || u.a0 >= nA ||
          u.b0 < u.a0 || u.b0 + u.n > rows_pad || u.a0 + GB_M > rows_pad) {
        std::printf("rows %d nA %d: tile (%d, %d) x %d\n", rows, nA, u.a0, u.b0, u.n);
        return 1;
      }
      by_tile[{u.a0, u.b0}].push_back(u);
    }
    // columns of each row tile: contiguous from its diagonal to the last column
    std::map<int, int> end;
    for (const auto& kv : by_tile) {
      const GbUnit& u = kv.second[0];
      if (!end.count(u.a0)) end[u.a0] = u.a0;
      if (end[u.a0] != u.b0) {
        std::printf("rows %d nA %d: row tile %d resumes at column %d, expected %d\n", rows, nA, u.a0, u.b0, end[u.a0]);
        return 1;
      }
      end[u.a0] = u.b0 + u.n;
      int64_t sum = 0, total = 0;
      for (const GbUnit& v : kv.second) {
        if (v.n != u.n || v.first < 0 || v.count <= 0 || v.first + (int64_t)v.count > n_stages) {
          std::printf("stages %d + %d of %d\n", v.first, v.count, n_stages);
          return 1;
        }
        total += v.count;
        for (int i = 0; i < v.count; ++i) sum += v.first + i;
      }
      // each slice once: their number and the sum of their positions
      if (total != n_stages || sum != (int64_t)n_stages * (n_stages - 1) / 2) {
        std::printf("tile (%d, %d): %lld stages of %d\n", u.a0, u.b0, (long long)total, n_stages);
        return 1;
      }
    }
    for (int a0 = 0; a0 < nA; a0 += GB_M)
      if (!end.count(a0) || end[a0] < rows) {
        std::printf("rows %d nA %d: row tile %d ends at %d\n", rows, nA, a0, end.count(a0) ? end[a0] : -1);
        return 1;
      }
  }
  std::printf("ok\n");
  return 0;
}
