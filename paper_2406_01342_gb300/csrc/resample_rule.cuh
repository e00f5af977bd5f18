// Which smaller image the w-plane transforms run on (resample.cu), and the taps that
// interpolate it. Host and device.
#pragma once

#include <algorithm>
#include <cmath>

namespace pc {

// Transforms on a smaller image of the same field.
struct Resample {
  int K = 0;            // interpolation taps (0: the transforms run on the image itself)
  int Nt = 0, G = 0;    // side of the transforms' image and of their grid
  double d = 1.0, beta = 0.0;
};

constexpr int RS_TERMS = 96;   // most terms of the window's power series (beta <= 63)

// The window's series: I0(beta sqrt(y)) / I0(beta) = sum_k c[k] y^k, all terms
// positive (c[k] = (beta / 2)^2k / k!^2 / I0(beta)).
struct Taps {
  double d;
  int N, Nt, K, terms;
  double c[RS_TERMS];
};

__host__ __device__ inline double tap_x(const Taps& t, int i) { return (i - t.N / 2) / t.d + t.Nt / 2; }
__host__ __device__ inline int tap_first(const Taps& t, int i) { return (int)floor(tap_x(t, i)) - t.K / 2 + 1; }

// sinpi(x): the caller's (device code has it as a function, host code has not)
__host__ __device__ inline double tap_weight(const Taps& t, double x, double sinpi_x) {
  const double z = x * (2.0 / t.K), y = 1.0 - z * z;
  if (!(y > 0.0)) return 0.0;
  const double s = fabs(x) < 1e-9 ? 1.0 : sinpi_x / (M_PI * x);
  double w = 0.0;
  for (int n = t.terms - 1; n >= 0; --n) w = fma(w, y, t.c[n]);
  return s * w;
}

inline Taps make_taps(const Resample& r, int N) {
  Taps t;
  t.d = r.d;
  t.N = N;
  t.Nt = r.Nt;
  t.K = r.K;
  double i0 = 0.0, term = 1.0;
  for (t.terms = 0; t.terms < RS_TERMS && (t.terms < 0.5 * r.beta || term > 1e-17 * i0); ++t.terms) {
    t.c[t.terms] = term;
    i0 += term;
    term *= 0.25 * r.beta * r.beta / ((double)(t.terms + 1) * (t.terms + 1));
  }
  for (int k = 0; k < t.terms; ++k) t.c[k] /= i0;
  return t;
}

// The smallest grid of side 512 or more whose image of side G / 2 still samples
// the visibilities: with K taps (16 .. 40) past the field's edge the pixels are d
// = N / (G / 2 - K) wide, and K must reach beta = 15.1. The small grid oversamples
// the pixels' field as much as the image's own grid does, up to 2.12: past that
// the planes cost more than the accuracy gives (1100 x 1100 at 2.05 / 2.12 / 2.3:
// errors 9.5e-7 / 6.7e-7 / 5.0e-7, against 7.2e-7 on the image's own grid; at 2.3 a
// quarter more planes). dl: the image's pixel, uv_max and w_max the largest |u| or
// |v| and |w|. The band holds the baseline and the slope w l / n of the w-term. The taps
// of a border pixel read samples further out, up to 1.19 times the field, where that
// slope is steeper: a band of the N x N pixels alone left errors of up to 1e-3
// there (4096 x 4096 over 5 degrees, turned by the w-term alone), one up to the smaller
// image's edge 5e-6, as a wave whose frequency climbs across the window is not
// held down by the window's own spectrum. With three times the climb such a wave is as
// good as one of constant frequency (2.1e-7 against 1.5e-7 at the least beta). In the
// configurations the w-term has 2 % of the turns and this moves nothing. Only grids of
// side 2048 and more are replaced: at 1024 the passes take 28 us of a 512 x 512
// certificate's 220, which the interpolation and a wider field's further w-planes would
// eat.
inline Resample choose_resample(int N, int G, double dl, double uv_max, double w_max) {
  Resample r;
  r.Nt = N;
  r.G = G;
  if (G < 2048) return r;
  const double half = 0.5 * N * dl;                       // half the image's field
  auto slope = [](double l) { return l / std::sqrt(1.0 - 2.0 * l * l); };   // of the w-term, at a corner
  const double sigma = std::min(2.12, (double)G / N);
  for (int g = 512; g < G; g *= 2)
    for (int K = 16; K <= 40; K += 8) {
      const double d = std::max((double)N / (g / 2 - K), sigma * N / g);
      const double h = 0.25 * g * d * dl;                 // half the smaller image's field
      if (d < 1.0 || 2.0 * h * h >= 1.0) continue;
      const double nu = d * dl * (uv_max + w_max * (slope(half) + 3.0 * (slope(h) - slope(half))));
      const double beta = M_PI * K * (0.5 - nu);
      if (beta < 15.1) continue;
      r.K = K;
      r.Nt = g / 2;
      r.G = g;
      r.d = d;
      r.beta = beta;
      return r;
    }
  return r;
}

// Rows of the two tables: the widest band of eight output rows. The kernel that applies
// them has shared memory for RS_MAX_WIDTH rows (894 at 4096 x 4096 with 40 taps on a grid
// of 512: (40 + 7) 4096 / 216 + 2).
constexpr int RS_MAX_WIDTH = 896;
inline void resample_widths(const Resample& r, int N, int* up, int* down) {
  Taps t;
  t.d = r.d;
  t.N = N;
  t.Nt = r.Nt;
  t.K = r.K;
  int wu = 0;
  for (int i = 0; i < N; i += 8) wu = std::max(wu, tap_first(t, std::min(i + 7, N - 1)) + r.K - tap_first(t, i));
  *up = wu + 1;   // the device may round a pixel that falls on a small one the other way
  // an input pixel i meets rows [first, first + K): those of eight rows span at
  // most (K + 7) d + 2 pixels
  *down = (int)std::ceil((r.K + 7) * r.d) + 2;
}

}  // namespace pc
