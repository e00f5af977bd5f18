// Host-side check of the smaller image that the rule chooses (resample_rule.cuh): a
// visibility's response on the smaller image, interpolated with the rule's taps,
// against its value at the N x N image's border and at pixels inside, in float64, for
// w-terms of none to nearly all of the turns and both signs. And the rows of its
// tables, over all sides and turns, against what the kernel has room for.
// Prints "ok" and exits 0, or the failures and exits 1.
#include "resample_rule.cuh"

#include <cstdio>
#include <vector>

using namespace pc;

static double response(double l, double m, double u, double v, double w) {
  const double r2 = l * l + m * m, n = std::sqrt(1.0 - r2);
  return std::cos(2.0 * M_PI * (u * l + v * m - w * r2 / (1.0 + n))) / n;
}

static double interpolated(const Taps& t, const std::vector<double>& small, int i, int j) {
  double wj[64], s = 0.0;
  const int ki = tap_first(t, i), kj = tap_first(t, j);
  for (int b = 0; b < t.K; ++b) {
    const double x = tap_x(t, j) - (kj + b);
    wj[b] = tap_weight(t, x, std::sin(M_PI * x));
  }
  for (int a = 0; a < t.K; ++a) {
    const double x = tap_x(t, i) - (ki + a), wi = tap_weight(t, x, std::sin(M_PI * x));
    double row = 0.0;
    for (int b = 0; b < t.K; ++b) row += wj[b] * small[(size_t)(ki + a) * t.Nt + kj + b];
    s += wi * row;
  }
  return s;
}

int main() {
  // two applications of taps that are within 1.5e-7 of a wave in the band, times 1 / n
  const double tol = 3e-7;
  const struct { int N; double fov_deg; } images[] = {{514, 2.0}, {600, 30.0}, {1100, 5.0}, {1100, 12.0}, {2048, 20.0},
                                                      {4096, 5.0}, {900, 50.0}};
  int bad = 0;
  for (const auto& im : images) {
    const double dl = im.fov_deg * M_PI / 180.0 / im.N, half = 0.5 * im.N * dl;
    const double slope = half / std::sqrt(1.0 - 2.0 * half * half);
    int G = 2048;
    while (G < 2 * im.N) G *= 2;
    for (double turns : {0.02, 0.08, 0.15, 0.19, 0.23, 0.3})        // per pixel at the image's corner
      for (double share : {0.0, 0.2, 0.5, 0.9, 1.0})                // of them from the w-term
        for (double sign : {1.0, -1.0}) {
          const double uv = (1.0 - share) * turns / dl, w = sign * share * turns / (dl * slope);
          const Resample r = choose_resample(im.N, G, dl, uv, std::fabs(w));
          if (r.K == 0) continue;
          const Taps t = make_taps(r, im.N);
          std::vector<double> small((size_t)r.Nt * r.Nt);
          for (int a = 0; a < r.Nt; ++a)
            for (int b = 0; b < r.Nt; ++b)
              small[(size_t)a * r.Nt + b] = response((a - r.Nt / 2) * dl * r.d, (b - r.Nt / 2) * dl * r.d, uv, -uv, w);
          double worst = 0.0;
          for (int e = 0; e < 600; ++e) {
            // corners, borders, inside
            const int k = (int)(((long long)e * 7919) % im.N), q = (int)(((long long)e * 104729) % im.N);
            const int i = e < 4 ? (e & 1 ? im.N - 1 : 0) : e % 3 == 0 ? 0 : e % 3 == 1 ? im.N - 1 : k;
            const int j = e < 4 ? (e & 2 ? im.N - 1 : 0) : q;
            const double l = (i - im.N / 2) * dl, m = (j - im.N / 2) * dl, n = std::sqrt(1.0 - l * l - m * m);
            worst = std::max(worst, n * std::fabs(interpolated(t, small, i, j) - response(l, m, uv, -uv, w)));
          }
          if (worst > tol) {
            std::printf("N %d, %g deg, %g turns, w %+g of them: G %d, K %d, error %.2e\n", im.N, im.fov_deg, turns,
                        sign * share, r.G, r.K, worst);
            bad = 1;
          }
        }
  }
  for (int N = 514; N <= 4096; N += 2) {
    int G = 2048;
    while (G < 2 * N) G *= 2;
    for (int e = 0; e <= 4000; ++e) {
      const double turns = 0.5 * e / 4000.0, dl = 0.05 / N;
      const Resample r = choose_resample(N, G, dl, turns / dl, 0.0);
      if (r.K == 0) continue;
      int up, down;
      resample_widths(r, N, &up, &down);
      if (up > RS_MAX_WIDTH || down > RS_MAX_WIDTH) {
        std::printf("N %d, %g turns: tables of %d and %d rows\n", N, turns, up, down);
        return 1;
      }
    }
  }
  if (!bad) std::printf("ok\n");
  return bad;
}
