// Plan construction: visibility binning by (gridding tile, w-plane), stable
// radix sort, sub-problem list, per-pixel kernel-correction table, workspace.
//
// The adjoint Phi* of Sect. 2.2 is evaluated as a type-1 non-uniform FFT
// (Sect. 5.2): each visibility is spread with an exponential-of-semicircle
// kernel of width W onto a 2x (or more) oversampled uv grid of side G, and
// onto P w-planes (w-stacking, the w-term of Sect. 2.1); every plane is
// inverse-FFT'd and the image is corrected for the kernel's Fourier transform,
// the w-screen and the 1/n factor.
//
// Geometry (all in FP64 here, once per plan):
//   g_u = frac(u dl) G  in [0, G)   grid coordinate in cells (the uv grid is G-periodic;
//   dl and G of the image that the planes are transformed on, see choose_resample)
//   x_w = (w - w0) / dw             plane coordinate
//   planes p = ceil(x_w - W/2) ... + W - 1, with dw <= 1 / (2 (s_max - s_min)),
//   s = n - 1 over that image, so that |dw (s - s_c)| <= 1/4 (oversampling 2 in w) on the N
//   x N pixels; up to 1/3 on the rim of a smaller image, which only the outer taps of
//   the interpolation read.
// Each visibility is replicated into every tile its W x W footprint touches
// (at most 2 x 2 tiles since W <= T), so a gridding CTA only ever reads the
// visibilities that touch its own tile.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "grid_win.cuh"
#include "pc_internal.cuh"

namespace pc {

// ------------------------------------------------------------------ host math

// Gauss-Legendre nodes and weights on [0, 1] (Newton on the Legendre recurrence).
static void gauss_legendre01(int n, std::vector<double>& x, std::vector<double>& w) {
  x.resize(n);
  w.resize(n);
  for (int i = 0; i < n; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5));
    double dp = 1.0;
    for (int it = 0; it < 100; ++it) {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
      double dz = p1 / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-16) break;
    }
    {
      double p0 = 1.0, p1 = z;
      for (int k = 2; k <= n; ++k) {
        double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      dp = n * (z * p1 - p0) / (z * z - 1.0);
    }
    x[i] = 0.5 * (1.0 + z);
    w[i] = 0.5 * 2.0 / ((1.0 - z * z) * dp * dp);
  }
}

// Fourier transform of the ES kernel in cell units at frequency t (cycles per cell):
//   psi(t) = int_{-W/2}^{W/2} phi(2y/W) e^{-j 2 pi y t} dy = W int_0^1 phi(z) cos(pi W z t) dz
// = W sum_q wphi[q] cos(pi wz[q] t) by quadrature (wz = W z_q, wphi = w_q phi(z_q)).
static double psi_hat_host(double t, int W, const std::vector<double>& wz, const std::vector<double>& wphi) {
  double s = 0.0;
  for (size_t q = 0; q < wz.size(); ++q) s += wphi[q] * std::cos(M_PI * wz[q] * t);
  return W * s;
}

// psi(k / G) for k <= n, the cosines by their three-term recurrence (n <= G / 4:
// its rounding stays below 1e-10).
static void psi_hat_grid(int n, int G, int W, const std::vector<double>& wz, const std::vector<double>& wphi,
                         std::vector<double>& out) {
  out.assign((size_t)n + 1, 0.0);
  for (size_t q = 0; q < wz.size(); ++q) {
    const double c1 = std::cos(M_PI * wz[q] / G);
    double c = 1.0, cm = c1;
    for (int k = 0; k <= n; ++k) {
      out[(size_t)k] += wphi[q] * c;
      const double cn = 2.0 * c1 * c - cm;
      cm = c;
      c = cn;
    }
  }
  for (double& v : out) v *= W;
}

// 1 / psi(t), |t| <= T, as a polynomial in y = 2 (t / T)^2 - 1: the w-kernel's
// correction, interpolated at Chebyshev nodes (psi is entire and even, its first
// zero past 0.7: 16 terms leave 1e-12 at T = 1/4 and 1e-10 at T = 0.4) and
// turned into powers of y for a Horner sum.
constexpr int kPsiTerms = 16;
static void psi_poly(double T, int W, const std::vector<double>& wz, const std::vector<double>& wphi, double* c) {
  double f[kPsiTerms];
  for (int i = 0; i < kPsiTerms; ++i) {
    const double y = std::cos(M_PI * (i + 0.5) / kPsiTerms);
    f[i] = 1.0 / psi_hat_host(T * std::sqrt(0.5 * (y + 1.0)), W, wz, wphi);
    c[i] = 0.0;
  }
  double prev[kPsiTerms] = {}, cur[kPsiTerms] = {1.0};   // powers of T_{k-1} and T_k
  for (int k = 0; k < kPsiTerms; ++k) {
    double v = 0.0;
    for (int i = 0; i < kPsiTerms; ++i) v += f[i] * std::cos(M_PI * k * (i + 0.5) / kPsiTerms);
    v *= (k ? 2.0 : 1.0) / kPsiTerms;
    for (int i = 0; i <= k; ++i) c[i] += v * cur[i];
    for (int i = std::min(k + 1, kPsiTerms - 1); i >= 0; --i) {   // T_{k+1} = 2 y T_k - T_{k-1} (T_1 = y)
      const double next = (k ? 2.0 : 1.0) * (i ? cur[i - 1] : 0.0) - prev[i];
      prev[i] = cur[i];
      cur[i] = next;
    }
  }
}

// ------------------------------------------------------------------ device kernels

// Order-preserving map of a double to uint64 (for atomic min / max).
__device__ __forceinline__ unsigned long long ordered_bits(double d) {
  unsigned long long b = (unsigned long long)__double_as_longlong(d);
  return (b & 0x8000000000000000ull) ? ~b : (b | 0x8000000000000000ull);
}

__global__ void k_uvw_scan(const double* __restrict__ uvw, int64_t M,
                           unsigned long long* wmin, unsigned long long* wmax, unsigned long long* uvmax,
                           int* bad) {
  unsigned long long lo = ~0ull, hi = 0ull, uv = 0ull;
  int nonfinite = 0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < M;
       k += (int64_t)gridDim.x * blockDim.x) {
    double u = uvw[3 * k], v = uvw[3 * k + 1], w = uvw[3 * k + 2];
    if (!isfinite(u) || !isfinite(v) || !isfinite(w)) nonfinite = 1;
    unsigned long long o = ordered_bits(w);
    lo = o < lo ? o : lo;
    hi = o > hi ? o : hi;
    // largest |u|, |v| (the bits of non-negative doubles order as integers)
    const unsigned long long m = (unsigned long long)__double_as_longlong(fmax(fabs(u), fabs(v)));
    uv = m > uv ? m : uv;
  }
  for (int off = 16; off; off >>= 1) {
    unsigned long long a = __shfl_xor_sync(0xffffffffu, lo, off);
    unsigned long long b = __shfl_xor_sync(0xffffffffu, hi, off);
    lo = a < lo ? a : lo;
    hi = b > hi ? b : hi;
    const unsigned long long c = __shfl_xor_sync(0xffffffffu, uv, off);
    uv = c > uv ? c : uv;
    nonfinite |= __shfl_xor_sync(0xffffffffu, nonfinite, off);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMin(wmin, lo);
    atomicMax(wmax, hi);
    atomicMax(uvmax, uv);
    if (nonfinite) atomicOr(bad, 1);
  }
}

// Bins: (tile, pair of plane starts ps >> 1); within a bin the slots are
// ordered by their tile-local row start b0 (then ps & 1). A sort key is
// bin << 7 | (b0 + 8) << 1 | (ps & 1), b0 in [-(W - 1), T - 1].
struct BinGeom {
  double dl, w0, dw, s_c;   // dl: pixel of the transforms' image
  double dl_pix;            // pixel of the image (the phases of atoms)
  int G, T, nT, W, P;
  int Pw;           // plane-start pairs (plane windows): ((P - W) >> 1) + 1, or 1 without w-stacking
  unsigned nbins;   // tiles x Pw
};
constexpr int kBinSubBits = 7;

__device__ __forceinline__ int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// Grid coordinate in cells of a baseline component: frac(u dl) G in [0, G).
__device__ __forceinline__ double turn_frac(double u, double dl) {
  const double U = u * dl;
  return U - rint(U);
}
__device__ __forceinline__ double grid_coord(double u, double dl, int G) {
  double g = turn_frac(u, dl) * G;
  if (g < 0.0) g += G;
  if (g >= G) g -= G;
  return g;
}

// Per visibility: fixed-point phase coefficients and up to 4 bin keys (one per
// tile touched by the footprint); unused key slots get the key nbins.
__global__ void k_vis_prep(const double* __restrict__ uvw, int64_t M, BinGeom g,
                           int4* __restrict__ vis_fx, unsigned* __restrict__ keys,
                           unsigned* __restrict__ ids) {
  int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= M) return;
  double u = uvw[3 * k], v = uvw[3 * k + 1], w = uvw[3 * k + 2];
  double gu = grid_coord(u, g.dl, g.G);
  double gv = grid_coord(v, g.dl, g.G);
  // 32-bit fixed-point turns of u dl and v dl (two's complement wrap = mod 1)
  int Ufx = (int)(unsigned)(long long)llrint(turn_frac(u, g.dl_pix) * 4294967296.0);
  int Vfx = (int)(unsigned)(long long)llrint(turn_frac(v, g.dl_pix) * 4294967296.0);
  float w_hi = (float)w;
  float w_lo = (float)(w - (double)w_hi);
  vis_fx[k] = make_int4(Ufx, Vfx, __float_as_int(w_hi), __float_as_int(w_lo));

  int a0 = (int)ceil(gu - 0.5 * g.W);
  int b0 = (int)ceil(gv - 0.5 * g.W);
  int ta0 = floor_div(a0, g.T), ta1 = floor_div(a0 + g.W - 1, g.T);
  int tb0 = floor_div(b0, g.T), tb1 = floor_div(b0 + g.W - 1, g.T);
  int ps = 0;
  if (g.P > 1) ps = min(max((int)ceil((w - g.w0) / g.dw - 0.5 * g.W), 0), g.P - g.W);
  for (int c = 0; c < 4; ++c) {
    int ta = ta0 + (c & 1), tb = tb0 + (c >> 1);
    unsigned key = g.nbins << kBinSubBits;
    if (ta <= ta1 && tb <= tb1) {
      int tu = ((ta % g.nT) + g.nT) % g.nT;
      int tv = ((tb % g.nT) + g.nT) % g.nT;
      const unsigned bin = (unsigned)((tv * g.nT + tu) * g.Pw + (ps >> 1));
      const unsigned b0l = (unsigned)(b0 - tb * g.T + 8);       // in [1, T + 7]
      key = (bin << kBinSubBits) | (b0l << 1) | (unsigned)(ps & 1);
    }
    keys[4 * k + c] = key;
    ids[4 * k + c] = (unsigned)(4 * k + c);
  }
}

// ---- stable LSD radix sort, 8-bit digits, 4096 keys per block

constexpr int RS_THREADS = 256;
constexpr int RS_ROUNDS = 16;
constexpr int RS_ITEMS = RS_THREADS * RS_ROUNDS;

__global__ void k_rs_hist(const unsigned* __restrict__ keys, int64_t n, int shift,
                          unsigned* __restrict__ hist, int nblk) {
  __shared__ unsigned h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  int64_t base = (int64_t)blockIdx.x * RS_ITEMS;
  for (int r = 0; r < RS_ROUNDS; ++r) {
    int64_t i = base + r * RS_THREADS + threadIdx.x;
    if (i < n) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
  }
  __syncthreads();
  hist[(int64_t)threadIdx.x * nblk + blockIdx.x] = h[threadIdx.x];
}

// Exclusive scan over the blocks of every digit's counts (block d: digit d), in
// place, and the digits' totals. The scatter adds up the totals itself. One block
// over all digits read 256 nblk entries through one SM: 2.5M entries and most of a
// 10M-visibility plan's 26 ms.
__global__ void __launch_bounds__(256) k_rs_scan(unsigned* __restrict__ hist, int nblk, unsigned* __restrict__ total) {
  __shared__ unsigned warp_tot[8];
  unsigned* row = hist + (int64_t)blockIdx.x * nblk;
  const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned run = 0;
  for (int base = 0; base < nblk; base += 256) {
    const int i = base + (int)threadIdx.x;
    const unsigned v = i < nblk ? row[i] : 0u;
    unsigned incl = v;
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= (unsigned)off) incl += t;
    }
    if (lane == 31) warp_tot[wid] = incl;
    __syncthreads();
    unsigned before = 0, all = 0;
    for (unsigned w = 0; w < 8; ++w) {
      before += w < wid ? warp_tot[w] : 0u;
      all += warp_tot[w];
    }
    if (i < nblk) row[i] = run + before + incl - v;
    run += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) total[blockIdx.x] = run;
}

__global__ void k_rs_scatter(const unsigned* __restrict__ kin, const unsigned* __restrict__ vin,
                             unsigned* __restrict__ kout, unsigned* __restrict__ vout, int64_t n,
                             int shift, const unsigned* __restrict__ hist, int nblk,
                             const unsigned* __restrict__ total) {
  __shared__ unsigned s_base[256];
  __shared__ unsigned s_tot[RS_THREADS / 32];
  __shared__ unsigned s_w[RS_THREADS / 32][256];
  int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  {
    // first position of digit tid: the totals of the digits before it
    const unsigned t = total[tid];
    unsigned incl = t;
    for (int off = 1; off < 32; off <<= 1) {
      const unsigned o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) s_tot[warp] = incl;
    __syncthreads();
    unsigned before = 0;
    for (int w = 0; w < warp; ++w) before += s_tot[w];
    s_base[tid] = before + incl - t + hist[(int64_t)tid * nblk + blockIdx.x];
  }
  int64_t base = (int64_t)blockIdx.x * RS_ITEMS;
  unsigned lt_mask = (1u << lane) - 1u;
  for (int r = 0; r < RS_ROUNDS; ++r) {
    for (int w = 0; w < RS_THREADS / 32; ++w) s_w[w][tid] = 0;
    __syncthreads();
    int64_t i = base + r * RS_THREADS + tid;
    bool valid = i < n;
    unsigned key = valid ? kin[i] : 0u;
    unsigned val = valid ? vin[i] : 0u;
    unsigned d = valid ? ((key >> shift) & 255u) : 256u;
    unsigned peers = __match_any_sync(0xffffffffu, d);
    unsigned rank = __popc(peers & lt_mask);
    if (valid && lane == __ffs(peers) - 1) s_w[warp][d] = __popc(peers);
    __syncthreads();
    unsigned run = 0;
    for (int w = 0; w < RS_THREADS / 32; ++w) {
      unsigned c = s_w[w][tid];
      s_w[w][tid] = run;
      run += c;
    }
    __syncthreads();
    if (valid) {
      unsigned pos = s_base[d] + s_w[warp][d] + rank;
      kout[pos] = key;
      vout[pos] = val;
    }
    __syncthreads();
    s_base[tid] += run;
  }
}

// off[b] = first sorted position whose bin is >= b, for b in [0, nbins]; the keys
// of unused slots (bin nbins) come last. A search per bin: one thread per key,
// filling the empty bins before it, left thousands to single threads.
__global__ void k_bin_offsets(const unsigned* __restrict__ keys, int64_t n, unsigned nbins,
                              int* __restrict__ off) {
  const unsigned b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b > nbins) return;
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((keys[mid] >> kBinSubBits) < b) lo = mid + 1; else hi = mid;
  }
  off[b] = (int)lo;
}

// Slot records in sorted order.
__global__ void k_slot_gather(const double* __restrict__ uvw, const unsigned* __restrict__ ids,
                              int64_t n_slots, BinGeom g, int2* __restrict__ slot_vis,
                              float4* __restrict__ slot_geom) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= n_slots) return;
  unsigned id = ids[j];
  int64_t k = id >> 2;
  int c = id & 3;
  double u = uvw[3 * k], v = uvw[3 * k + 1], w = uvw[3 * k + 2];
  double gu = grid_coord(u, g.dl, g.G);
  double gv = grid_coord(v, g.dl, g.G);
  int a0 = (int)ceil(gu - 0.5 * g.W);
  int b0 = (int)ceil(gv - 0.5 * g.W);
  int ta = floor_div(a0, g.T) + (c & 1);
  int tb = floor_div(b0, g.T) + (c >> 1);
  int a0l = a0 - ta * g.T;   // footprint start relative to the tile, in [-W+1, T-1]
  int b0l = b0 - tb * g.T;
  float xw = 0.0f, tau = 0.0f;
  int ps = 0;
  if (g.P > 1) {
    double x = (w - g.w0) / g.dw;
    ps = min(max((int)ceil(x - 0.5 * g.W), 0), g.P - g.W);
    xw = (float)(x - ps);
    double tt = (w - g.w0) * g.s_c;     // pre-twiddle e^{j 2 pi (w - w0) s_c}, in turns
    tau = (float)(tt - rint(tt));
  }
  slot_vis[j] = make_int2((int)k, (int)((unsigned)(a0l + 64) | ((unsigned)(b0l + 64) << 8) | ((unsigned)ps << 16)));
  slot_geom[j] = make_float4((float)(gu - a0), (float)(gv - b0), xw, tau);
}

struct PixGeom {
  double dl, w0, dw, s_c, inv_t;   // inv_t: 1 / T of psi_poly
  int N, W;
  bool wstack;
};

// Per-pixel tables are even in the pixel's offsets i' = i - N/2, j' = j - N/2: a
// thread per quadrant pixel evaluates its FP64 square root and divisions (a slow
// pipe on this GPU) once and writes the up to four pixels (+-i', +-j').
template <class T, class F>
__device__ __forceinline__ void write_quadrant(T* __restrict__ out, int N, int a, int b, F value) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int ip = q & 2 ? -a : a, jp = q & 1 ? -b : b;
    if ((q & 2 && a == 0) || (q & 1 && b == 0) || ip >= N / 2 || jp >= N / 2) continue;
    out[(size_t)(ip + N / 2) * N + (jp + N / 2)] = value(ip, jp);
  }
}

// Epilogue coefficients: {Re, Im} of e^{j 2 pi w0 s} / (n psi(i') psi(j') psi_w(t))
// and t = dw (s - s_c) as a double-float (hi, lo). rpsi: 1 / psi(k / G), k <= N/2;
// poly: 1 / psi_w(t) (psi_poly).
__global__ void k_pix_tab(PixGeom g, const double* __restrict__ rpsi, const double* __restrict__ poly,
                          float4* __restrict__ out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x, a = blockIdx.y;
  if (b > g.N / 2) return;
  const double l = a * g.dl, m = b * g.dl;
  const double r2 = l * l + m * m, q = 1.0 - r2;
  // 1 / n = q^(-1/2) and 1 / (1 + n): an FP32 value and one Newton step each (1e-13
  // relative). n - 1 = -r2 / (1 + n) keeps that accuracy; the difference q / n - 1 was off
  // by 5e-14, which |w| multiplies into turns
  double rn = (double)rsqrtf((float)q);
  rn *= fma(-0.5 * q * rn, rn, 1.5);
  const double n1 = fma(q, rn, 1.0);
  double rn1 = (double)(1.f / (float)n1);
  rn1 *= fma(-n1, rn1, 2.0);
  const double s = -r2 * rn1;        // n - 1
  double t = 0.0, rw = 1.0;
  if (g.wstack) {
    t = g.dw * (s - g.s_c);
    const double z = t * g.inv_t, y = 2.0 * z * z - 1.0;
    rw = poly[kPsiTerms - 1];
#pragma unroll
    for (int k = kPsiTerms - 2; k >= 0; --k) rw = fma(rw, y, poly[k]);
  }
  double ct = g.w0 * s;
  ct -= rint(ct);                    // exact reduction to [-1/2, 1/2] turns in FP64
  float snf, csf;                    // then an FP32 sine / cosine (~1e-7): FP64 ones are slow here
  sincospif(2.0f * (float)ct, &snf, &csf);
  const double d = rpsi[a] * rpsi[b] * rw * rn;
  const float t_hi = (float)t;
  const float4 v = make_float4((float)((double)csf * d), (float)((double)snf * d), t_hi, (float)(t - (double)t_hi));
  write_quadrant(out, g.N, a, b, [&](int, int) { return v; });
}

// Per-pixel unit-weight atoms, evaluated once per plan; the solver's
// per-iteration bookkeeping then only gathers them.
__global__ void k_atom_tab(int N, double dl, float4* __restrict__ out) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x, a = blockIdx.y;
  if (b > N / 2) return;
  // pixel (-a, -b) exists for every a, b <= N/2
  const float4 at = make_atom((N / 2 - a) * N + (N / 2 - b), 1.f, false, N, dl);
  write_quadrant(out, N, a, b, [&](int ip, int jp) {
    return make_float4(__int_as_float((int)(((unsigned)ip << 16) | ((unsigned)jp & 0xffffu))), at.y, at.z, at.w);
  });
}

// FFT twiddle tables: tw[k] = e^{+2 pi i k / G}; tw2 [k1 < G/32][l < 32] of the
// one-warp FFT (G = 512, 1024); tw_in [k1 < 16][l < 32] and tw_big [k1 < G/512][n'
// < 512] of the one-CTA FFT (G >= 2048). Null tables are left out.
__global__ void k_twiddles(int G, float2* __restrict__ tw, float2* __restrict__ tw2, float2* __restrict__ tw_in,
                           float2* __restrict__ tw_big) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= G) return;
  auto root = [&](int e) {
    double sn, cs;
    sincospi(2.0 * (e % G) / G, &sn, &cs);
    return make_float2((float)cs, (float)sn);
  };
  tw[k] = root(k);
  if (tw2) tw2[k] = root((k >> 5) * (k & 31));                       // G entries
  if (tw_in && k < 512) tw_in[k] = root((k >> 5) * (k & 31) * (G / 512));
  if (tw_big) tw_big[k] = root((k >> 9) * (k & 511));
}

// The stream plan construction runs on: plan buffers come from the library's
// pool ordered on it (construction ends with a synchronisation of this stream,
// after which every stream may use them).
static thread_local cudaStream_t g_build_stream = nullptr;

static int dev_alloc(pc_plan_s* p, void** ptr, size_t bytes) {
  PC_TRY(dmalloc(ptr, bytes == 0 ? 16 : bytes, g_build_stream));
  p->owned.push_back(*ptr);
  return PC_OK;
}

template <class T>
static int dev_alloc_t(pc_plan_s* p, T** ptr, size_t count) {
  return dev_alloc(p, reinterpret_cast<void**>(ptr), count * sizeof(T));
}

// Host arrays on their way to or from the device, in recycled pinned memory, so
// that a copy neither waits for the stream nor for the host array's lifetime (a
// copy from pageable memory waits for the stream first: thirteen of them kept host
// and device taking turns). Chunks of powers of two, so that plans of other sizes
// reuse them; released after the stream has been waited for.
struct Staging {
  std::vector<void*> chunks;
  char* at = nullptr;
  size_t left = 0;
  cudaStream_t st = nullptr;
  ~Staging() {
    if (!chunks.empty()) cudaStreamSynchronize(st);
    for (void* q : chunks) pinned_put(q);
  }
  void* block(size_t bytes) {
    bytes = (bytes + 15) / 16 * 16;
    if (bytes > left) {
      size_t chunk = 256 * 1024;
      while (chunk < bytes) chunk *= 2;
      void* q = pinned_get(chunk);
      if (!q) return nullptr;
      chunks.push_back(q);
      at = static_cast<char*>(q);
      left = chunk;
    }
    void* q = at;
    at += bytes;
    left -= bytes;
    return q;
  }
  int upload(void* dst, const void* src, size_t bytes) {
    if (bytes == 0) return PC_OK;
    void* q = block(bytes);
    if (!q) return fail(PC_ERR_OOM, "plan: %zu bytes of pinned memory", bytes);
    std::memcpy(q, src, bytes);
    PC_CUDA(cudaMemcpyAsync(dst, q, bytes, cudaMemcpyHostToDevice, st));
    return PC_OK;
  }
};

// Temporary device buffers of plan construction, freed on every exit path.
struct TmpBufs {
  std::vector<void*> v;
  cudaStream_t st = nullptr;
  ~TmpBufs() {
    for (void* q : v) dfree(q, st);   // ordered after their last use on st
  }
  int alloc(void** ptr, size_t bytes) {
    PC_TRY(dmalloc(ptr, bytes == 0 ? 16 : bytes, st));
    v.push_back(*ptr);
    return PC_OK;
  }
};

// Splits every (tile, plane group) slot range into equal pieces of at most
// `piece` slots (multiples of 64, the tensor-core stage) and uploads the list.
// Window CTAs: a tile whose slots exceed `cap` is split into equal parts
// (each part takes its share of every plane window of the tile); heaviest
// CTAs first, so the last wave holds the light ones.
static int split_win_parts(pc_plan_s* p, int cap, int4* dst, int* n_out, Staging& up) {
  cap = std::max(cap, 64);
  std::vector<int4> subs;
  for (const int2& t : p->win_tiles) {
    const int parts = ceil_div(t.y, cap);
    for (int k = 0; k < parts; ++k) subs.push_back(make_int4(t.x, k, parts, ceil_div(t.y, parts)));
  }
  std::stable_sort(subs.begin(), subs.end(), [](const int4& a, const int4& b) { return a.w > b.w; });
  if ((int64_t)subs.size() > p->wsub_cap) return fail(PC_ERR_CAPACITY, "plan: %zu window CTAs", subs.size());
  *n_out = (int)subs.size();
  return up.upload(dst, subs.data(), sizeof(int4) * subs.size());
}

// The window gridding's CTAs (each part adds its tile to the grid).
static int split_wsubs(pc_plan_s* p, int cap, Staging& up) {
  PC_TRY(split_win_parts(p, cap, p->wsubs, &p->n_wsub, up));
  p->win_cap = std::max(cap, 64);
  return PC_OK;
}

// The window degridding's CTAs (each part reads its tile's planes; no part
// writes the grid, so the split only costs plane loads).
static int split_dwsubs(pc_plan_s* p, int cap, Staging& up) {
  PC_TRY(split_win_parts(p, cap, p->dwsubs, &p->n_dwsub, up));
  p->dwin_cap = std::max(cap, 64);
  return PC_OK;
}

static int split_subs(pc_plan_s* p, int piece, Staging& up) {
  std::vector<int4> subs;
  const int stage = p->wstack ? 64 : 32;   // the tensor-core stage; k_grid's smallest
  for (const int4& r : p->sub_ranges) {
    const int len = r.w - r.z;
    const int n_pieces = ceil_div(len, piece);
    const int sz = ceil_div(ceil_div(len, n_pieces), stage) * stage;
    for (int s = r.z; s < r.w; s += sz) subs.push_back(make_int4(r.x, r.y, s, std::min(r.w, s + sz)));
  }
  if ((int)subs.size() > p->sub_cap) return fail(PC_ERR_CAPACITY, "plan: %zu sub-problems", subs.size());
  p->n_sub = (int)subs.size();
  p->grid_piece = piece;
  return up.upload(p->subs, subs.data(), sizeof(int4) * subs.size());
}

__global__ void k_fill_ones(float2* __restrict__ h, int64_t M) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < M; k += (int64_t)gridDim.x * blockDim.x)
    h[k] = make_float2(1.0f, 0.5f);
}

// Median of `reps` timed calls of f (after one untimed call), in microseconds.
template <class F>
static int time_us(cudaStream_t st, int reps, F f, double* out) {
  cudaEvent_t a, b;
  PC_CUDA(cudaEventCreate(&a));
  PC_CUDA(cudaEventCreate(&b));
  std::vector<double> t;
  int rc = f();
  for (int i = 0; i < reps && rc == PC_OK; ++i) {
    cudaEventRecord(a, st);
    rc = f();
    cudaEventRecord(b, st);
    cudaEventSynchronize(b);
    float ms = 0.f;
    cudaEventElapsedTime(&ms, a, b);
    t.push_back(1e3 * ms);
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  PC_TRY(rc);
  std::sort(t.begin(), t.end());
  *out = t[t.size() / 2];
  return PC_OK;
}

// Plan-time autotuner: times, on this plan's binned visibilities, the
// gridding kernels (tensor cores vs CUDA cores, w-stacked plans) x the
// sub-problem sizes, then the first FFT pass's rows per CTA, and keeps the
// fastest of each.
static int autotune(pc_plan_s* p, cudaStream_t st) {
  if (p->M <= 0 || p->n_sub == 0) return PC_OK;
  Staging up;
  up.st = st;
  k_fill_ones<<<(int)std::min<int64_t>(4096, (p->M + 255) / 256), 256, 0, st>>>(p->resid, p->M);
  PC_LAUNCH_CHECK();
  const int user_mode = p->grid_mode;
  std::vector<int> modes = {user_mode};
  if (user_mode == 0 && p->wstack) modes = p->W <= 7 ? std::vector<int>{3, 2, 1} : std::vector<int>{2, 1};
  double best = 1e300;
  int best_mode = user_mode, best_piece = grid_win_mode(p) ? p->win_cap : p->grid_piece;
  for (int mode : modes) {
    p->grid_mode = mode;
    const bool win = grid_win_mode(p);
    // window gridding: slots per CTA before a tile is split; else the sub-problem size
    const std::vector<int> pieces = win ? std::vector<int>{p->win_cap, 1024, 4096, 16384, 65536}
                                        : std::vector<int>{256, 512, 1024, 2048, 4096};
    for (int piece : pieces) {
      p->grid_mode = mode;
      PC_TRY(win ? split_wsubs(p, piece, up) : split_subs(p, piece, up));
      double us = 0.0;
      PC_TRY(time_us(st, 3, [&] { return launch_grid(p, p->resid, st); }, &us));
      if (us < best) {
        best = us;
        best_mode = mode;
        best_piece = piece;
      }
    }
  }
  p->grid_mode = best_mode;
  PC_TRY(grid_win_mode(p) ? split_wsubs(p, best_piece, up) : split_subs(p, best_piece, up));
  p->tune_grid_us = best;
  PC_TRY(launch_grid(p, p->resid, st));         // a gridded plane set for the FFT timing
  // first pass: the one-warp register FFT (where G allows it) against the
  // shared-memory Stockham kernel at each rows-per-CTA
  double best_fft = 1e300;
  int best_R = 0, best_rw = 0;
  p->fft_warp = 1;
  if (fft_rows_warp(p) || fft_rows_big(p)) {
    PC_TRY(time_us(st, 3, [&] { return launch_fft_rows(p, st); }, &best_fft));
    best_rw = 1;
  }
  p->fft_warp = 0;
  for (int R : {1, 2, 4, 8, 16, 32}) {
    if (((size_t)2 * R * (p->G + 1) + p->G) * sizeof(float2) > 200 * 1024) break;
    p->fft_R = R;
    double us = 0.0;
    PC_TRY(time_us(st, 3, [&] { return launch_fft_rows(p, st); }, &us));
    if (us < best_fft) {
      best_fft = us;
      best_R = R;
      best_rw = 0;
    }
  }
  p->fft_R = best_R;
  p->tune_fft_us = best_fft;
  p->fft_warp = best_rw;
  // second pass: one-warp register FFTs against the Stockham kernel at each
  // number of planes transformed together (shared memory vs CTAs per SM)
  PC_TRY(launch_fft_rows(p, st));
  double best_cols = 1e300;
  int best_pg = 1, best_cw = 0;
  p->fft_warp = best_rw | 2;
  if (fft_cols_warp(p) || fft_cols_big(p)) {
    PC_TRY(time_us(st, 3, [&] { return launch_fft_cols_epilogue(p, p->mu, 1.0f, nullptr, st); },
                   &best_cols));
    best_cw = 2;
  }
  p->fft_warp = best_rw;
  for (int pg : {1, 2, 4, 8}) {
    p->fft_cols_pg = pg;
    if (cols_planes_per_pass(p) != pg) break;   // beyond the planes or shared memory
    double us = 0.0;
    PC_TRY(time_us(st, 3, [&] { return launch_fft_cols_epilogue(p, p->mu, 1.0f, nullptr, st); }, &us));
    if (us < best_cols) {
      best_cols = us;
      best_pg = pg;
      best_cw = 0;
    }
  }
  p->fft_cols_pg = best_pg;
  p->tune_fft_cols_us = best_cols;
  p->fft_warp = best_rw | best_cw;
  // window degridding: slots per CTA before a tile is split (into the
  // residual buffer, cleared below; the grid holds the planes timed above)
  if (grid_win_mode(p)) {
    double best_dw = 1e300;
    int best_cap = p->dwin_cap;
    for (int cap : {p->dwin_cap, 2048, 4096, 8192, 16384}) {
      PC_TRY(split_dwsubs(p, cap, up));
      double us = 0.0;
      PC_TRY(time_us(st, 3, [&] { return launch_degrid_win(p, p->resid, st); }, &us));
      if (us < best_dw) {
        best_dw = us;
        best_cap = cap;
      }
    }
    PC_TRY(split_dwsubs(p, best_cap, up));
    p->tune_degrid_us = best_dw;
  }
  p->tuned = true;
  PC_CUDA(cudaMemsetAsync(p->resid, 0, sizeof(float2) * p->M, st));
  PC_CUDA(cudaStreamSynchronize(st));
  return PC_OK;
}

static int build_plan(pc_plan_s* p, const double* uvw, cudaStream_t st, int max_planes) {
  const int64_t M = p->M;
  const int N = p->N;
  g_build_stream = st;
  TmpBufs tmp;
  tmp.st = st;
  Staging up;
  up.st = st;

  // ---- w range, largest |u|, |v| and finiteness
  double uv_max = 0.0;
  if (M > 0) {
    unsigned long long* dmm;
    int* dbad;
    PC_TRY(tmp.alloc((void**)&dmm, 3 * sizeof(unsigned long long) + sizeof(int) * 2));
    dbad = reinterpret_cast<int*>(dmm + 3);
    PC_CUDA(cudaMemsetAsync(dmm, 0xff, sizeof(unsigned long long), st));
    PC_CUDA(cudaMemsetAsync(dmm + 1, 0, 2 * sizeof(unsigned long long) + 2 * sizeof(int), st));
    int blocks = (int)std::min<int64_t>(4096, (M + 255) / 256);
    k_uvw_scan<<<blocks, 256, 0, st>>>(uvw, M, dmm, dmm + 1, dmm + 2, dbad);
    PC_LAUNCH_CHECK();
    struct { unsigned long long mm[3]; int bad[2]; } got;
    PC_CUDA(cudaMemcpyAsync(&got, dmm, sizeof(got), cudaMemcpyDeviceToHost, st));
    PC_CUDA(cudaStreamSynchronize(st));
    const unsigned long long* hmm = got.mm;
    if (got.bad[0]) return fail(PC_ERR_INVALID_ARG, "plan: uvw contains NaN or Inf");
    auto unmap = [](unsigned long long o) {
      unsigned long long b = (o & 0x8000000000000000ull) ? (o & 0x7fffffffffffffffull) : ~o;
      double d;
      std::memcpy(&d, &b, sizeof(d));
      return d;
    };
    p->w_min = unmap(hmm[0]);
    p->w_max = unmap(hmm[1]);
    std::memcpy(&uv_max, &hmm[2], sizeof(uv_max));
  }

  // ---- geometry
  p->G_image = 32;
  while (p->G_image < 2 * N) p->G_image *= 2;
  p->dl = p->fov / N;
  p->Nt = N;
  p->G = p->G_image;
  {
    // corner of the image; the transforms' smaller one reaches a little further
    const double half = 0.5 * N * p->dl, r2 = 2.0 * half * half;
    const double w_abs = std::max(std::fabs(p->w_min), std::fabs(p->w_max));
    // one plane's transforms are a few per cent of a call, and without a w-term's error
    // that of a smaller grid shows (dirty images, own grid and smaller: 1462 x 1462, 1.2M
    // 2.0e-7 and 2.5e-7, 459 and 457 us; 4096 x 4096, 10M 2.6e-7 and 4.1e-7, 3320 and 3170
    // us; forward at 1462 80 and 89 us)
    if (M > 0 && p->w_max > p->w_min && p->fft_warp != 0 && r2 < 0.4)
      p->resample = choose_resample(N, p->G_image, p->dl, uv_max, w_abs);
    if (p->resample.K > 0) {
      // its wider field takes more w-planes: not beyond the caller's cap
      const double h = 0.5 * p->resample.Nt * p->dl * p->resample.d, r2t = 2.0 * h * h;
      const double s_range = r2t / (1.0 + std::sqrt(1.0 - r2t));
      if (std::ceil((p->w_max - p->w_min) * 2.0 * s_range) + p->W > max_planes) p->resample.K = 0;
    }
    if (p->resample.K > 0) {
      p->Nt = p->resample.Nt;
      p->G = p->resample.G;
    }
  }
  const int Nt = p->Nt;
  const double dlt = p->resample.K > 0 ? p->dl * p->resample.d : p->dl;
  p->logG = 0;
  while ((1 << p->logG) < p->G) ++p->logG;
  p->nT = p->G / p->T;
  // the kernel's shape: 2.30 W suits an oversampling of 2; a smaller image's is a
  // little more (pi (1 - 1 / 2 sigma) W, as for that 2.30)
  p->beta = 2.30 * p->W;
  if (p->resample.K > 0)
    p->beta = 0.976 * M_PI * (1.0 - 0.5 / std::min(2.3, p->resample.G * p->resample.d / N)) * p->W;
  const double half = 0.5 * Nt * dlt;
  const double r2c = 2.0 * half * half;
  const double s_min = -r2c / (1.0 + std::sqrt(1.0 - r2c));
  const double s_max = 0.0;
  // The planes are spaced for the corner of the transforms' image but centred on the
  // N x N pixels' own range, which then is sampled more finely than at 2; only the
  // rim that the interpolation's outer taps touch lies beyond 1/4 (figures at
  // choose_resample).
  const double half_n = 0.5 * N * p->dl, r2n = 2.0 * half_n * half_n;
  const double s_min_n = -r2n / (1.0 + std::sqrt(1.0 - r2n));
  double t_max = 0.25;
  p->phase = phase_scale(std::max(std::fabs(p->w_min), std::fabs(p->w_max)), -s_min);
  if (M > 0 && p->w_max > p->w_min) {
    p->wstack = true;
    p->dw = 1.0 / (2.0 * (s_max - s_min));
    long long planes = (long long)std::ceil((p->w_max - p->w_min) / p->dw) + p->W;
    if (planes > max_planes)
      return fail(PC_ERR_INVALID_ARG, "plan: %lld w-planes needed, max_planes is %d", planes,
                  max_planes);
    // A visibility meets W planes from the first one at or past its footprint's start, so
    // a range of r plane spacings needs floor(r) + 1 starts where they are placed for it
    // (from the first start exactly at w_min it took one more: 9 planes for r = 1.02,
    // two groups in the tensor-core gridding instead of one: 136 -> 93 us for 200k
    // visibilities, 45 -> 19 us in the second FFT pass). What r lacks to the next whole
    // number the spacing gives up, by half at most, which lowers the w-kernel's aliasing
    // at no cost.
    double r = (p->w_max - p->w_min) / p->dw;
    const int starts = std::max(1, (int)std::floor(r)) + 1;
    const double fuller = std::min(starts - 0.02, 2.0 * r);
    if (fuller > r) {
      p->dw *= r / fuller;
      r = fuller;
    }
    p->P = starts - 1 + p->W;
    p->w0 = p->w_min - (0.5 * p->W + 0.5 * (starts - r) - 1.0) * p->dw;
    p->s_c = 0.5 * (s_min_n + s_max);
    t_max = std::max(p->dw * std::max(p->s_c - s_min, s_max - p->s_c), 0.25);
  } else {
    p->wstack = false;
    p->P = 1;
    p->dw = 1.0;
    p->w0 = M > 0 ? p->w_min : 0.0;
    p->s_c = 0.0;
  }
  {
    int ngroups = ceil_div(p->P, 8);      // gridding keeps <= 8 planes of a tile in registers
    p->Qg = ceil_div(p->P, ngroups);
  }

  // ---- tables: ES transform, twiddles, per-pixel corrections
  std::vector<double> gx, gw;
  gauss_legendre01(kGlNodes, gx, gw);
  // node factors of the quadrature: W z_q and w_q phi(z_q)
  std::vector<double> wz(kGlNodes), wphi(kGlNodes);
  for (int q = 0; q < kGlNodes; ++q) {
    wz[q] = p->W * gx[q];
    wphi[q] = gw[q] * std::exp(p->beta * (std::sqrt(std::max(0.0, 1.0 - gx[q] * gx[q])) - 1.0));
  }
  std::vector<double> rpsi;
  psi_hat_grid(Nt / 2, p->G, p->W, wz, wphi, rpsi);
  for (double& v : rpsi) v = 1.0 / v;
  rpsi.resize(rpsi.size() + kPsiTerms);
  double* poly = rpsi.data() + Nt / 2 + 1;
  psi_poly(t_max, p->W, wz, wphi, poly);
  double* d_psi;
  PC_TRY(tmp.alloc((void**)&d_psi, sizeof(double) * rpsi.size()));
  PC_TRY(up.upload(d_psi, rpsi.data(), sizeof(double) * rpsi.size()));
  const int64_t NN = (int64_t)N * N, NNt = (int64_t)Nt * Nt;
  PC_TRY(dev_alloc_t(p, &p->pix_tab, NNt));
  {
    PixGeom pg{dlt, p->w0, p->dw, p->s_c, 1.0 / t_max, Nt, p->W, p->wstack};
    k_pix_tab<<<dim3(ceil_div(Nt / 2 + 1, 128), Nt / 2 + 1), 128, 0, st>>>(pg, d_psi, d_psi + Nt / 2 + 1, p->pix_tab);
    PC_LAUNCH_CHECK();
  }
  PC_TRY(dev_alloc_t(p, &p->atom_tab, NN));
  k_atom_tab<<<dim3(ceil_div(N / 2 + 1, 128), N / 2 + 1), 128, 0, st>>>(N, p->dl, p->atom_tab);
  PC_LAUNCH_CHECK();
  if (p->resample.K > 0) {
    resample_widths(p->resample, N, &p->up.width, &p->down.width);
    const int gu = ceil_div(N, 8), gd = ceil_div(Nt, 8);
    PC_TRY(dev_alloc_t(p, &p->up.first, (size_t)gu));
    PC_TRY(dev_alloc_t(p, &p->up.w, (size_t)gu * p->up.width * 8));
    PC_TRY(dev_alloc_t(p, &p->down.first, (size_t)gd));
    PC_TRY(dev_alloc_t(p, &p->down.w, (size_t)gd * p->down.width * 8));
    PC_TRY(dev_alloc_t(p, &p->small_img, (size_t)NNt));
    PC_TRY(dev_alloc_t(p, &p->small_tmp, (size_t)Nt * N));
    PC_TRY(fill_band_tables(p->resample, N, &p->up, &p->down, st));
  }
  PC_TRY(dev_alloc_t(p, &p->twiddle, p->G));
  if (p->G == 512 || p->G == 1024) PC_TRY(dev_alloc_t(p, &p->tw2, p->G));
  if (fft_big_size(p->G)) {
    PC_TRY(dev_alloc_t(p, &p->tw_in, 512));
    PC_TRY(dev_alloc_t(p, &p->tw_big, p->G));
  }
  k_twiddles<<<ceil_div(p->G, 128), 128, 0, st>>>(p->G, p->twiddle, p->tw2, p->tw_in, p->tw_big);
  PC_LAUNCH_CHECK();

  // ---- workspaces
  PC_TRY(dev_alloc_t(p, &p->grid, (size_t)p->P * p->G * p->G));
  // only the Stockham passes read cells that no visibility reaches (whole rows of
  // the grid, whole columns of their transposed output): those stay zero from here
  const bool whole_rows = !(p->G == 512 || p->G == 1024 || fft_big_size(p->G)) || p->fft_warp == 0 || p->want_tune;
  if (whole_rows) PC_CUDA(cudaMemsetAsync(p->grid, 0, sizeof(float2) * (size_t)p->P * p->G * p->G, st));
  // the Stockham passes' transposed pass-1 output (every G up to 1024; for
  // larger grids only when those passes can be chosen: forced, or timed by
  // the autotuner; the one-CTA passes use the compact buffer xc instead)
  if (!fft_big_size(p->G) || p->fft_warp == 0 || p->want_tune) {
    PC_TRY(dev_alloc_t(p, &p->fft1, (size_t)p->P * Nt * p->G));
    if (whole_rows) PC_CUDA(cudaMemsetAsync(p->fft1, 0, sizeof(float2) * (size_t)p->P * Nt * p->G, st));
  }
  PC_TRY(dev_alloc_t(p, &p->resid, (size_t)std::max<int64_t>(M, 1)));
  PC_TRY(dev_alloc_t(p, &p->mu, (size_t)NN));
  PC_TRY(dev_alloc_t(p, &p->mark, (size_t)NN));
  PC_CUDA(cudaMemsetAsync(p->mark, 0, NN, st));
  PC_TRY(dev_alloc_t(p, &p->dscal, sizeof(Scalars) / sizeof(double)));
  p->uscal = reinterpret_cast<unsigned*>(p->dscal + 8);
  p->iscal = reinterpret_cast<int32_t*>(p->uscal + 8);
  PC_CUDA(cudaMemsetAsync(p->iscal, 0, 8 * sizeof(int32_t), st));
  p->sel_blocks_n = ceil_div(NN, kSelItems);
  PC_TRY(dev_alloc_t(p, &p->sel_blocks, (size_t)p->sel_blocks_n + 2));
  PC_CUDA(cudaMemsetAsync(p->sel_blocks, 0, sizeof(int32_t) * ((size_t)p->sel_blocks_n + 2), st));
  PC_TRY(dev_alloc_t(p, &p->vis_fx, (size_t)std::max<int64_t>(M, 1)));

  if (M == 0) {
    p->n_slots = 0;
    p->n_sub = 0;
    PC_TRY(dev_alloc_t(p, &p->slot_vis, 1));
    PC_TRY(dev_alloc_t(p, &p->slot_geom, 1));
    PC_TRY(dev_alloc_t(p, &p->subs, 1));
    PC_CUDA(cudaStreamSynchronize(st));
    return PC_OK;
  }

  // ---- binning keys
  p->Pw = p->wstack ? ((p->P - p->W) >> 1) + 1 : 1;
  const unsigned nbins = (unsigned)((int64_t)p->nT * p->nT * p->Pw);
  if ((int64_t)p->nT * p->nT * p->Pw >= (1ll << (32 - kBinSubBits)))
    return fail(PC_ERR_INVALID_ARG, "plan: too many (tile, plane pair) bins");
  const int64_t nkeys = 4 * M;
  unsigned *k0, *k1, *v0, *v1, *hist;
  int* off;
  PC_TRY(tmp.alloc((void**)&k0, sizeof(unsigned) * nkeys));
  PC_TRY(tmp.alloc((void**)&k1, sizeof(unsigned) * nkeys));
  PC_TRY(tmp.alloc((void**)&v0, sizeof(unsigned) * nkeys));
  PC_TRY(tmp.alloc((void**)&v1, sizeof(unsigned) * nkeys));
  const int nblk = ceil_div(nkeys, RS_ITEMS);
  PC_TRY(tmp.alloc((void**)&hist, sizeof(unsigned) * 256 * ((size_t)nblk + 1)));
  unsigned* const total = hist + 256 * (size_t)nblk;
  PC_TRY(tmp.alloc((void**)&off, sizeof(int) * ((size_t)nbins + 1)));
  BinGeom bg{dlt, p->w0, p->dw, p->s_c, p->dl, p->G, p->T, p->nT, p->W, p->P, p->Pw, nbins};
  k_vis_prep<<<ceil_div(M, 256), 256, 0, st>>>(uvw, M, bg, p->vis_fx, k0, v0);
  PC_LAUNCH_CHECK();

  // ---- stable radix sort of the keys (values = slot ids)
  int nbits = 1;
  while ((1ull << nbits) <= ((unsigned long long)nbins << kBinSubBits)) ++nbits;
  unsigned *kin = k0, *vin = v0, *kout = k1, *vout = v1;
  for (int shift = 0; shift < nbits; shift += 8) {
    k_rs_hist<<<nblk, RS_THREADS, 0, st>>>(kin, nkeys, shift, hist, nblk);
    PC_LAUNCH_CHECK();
    k_rs_scan<<<256, 256, 0, st>>>(hist, nblk, total);
    PC_LAUNCH_CHECK();
    k_rs_scatter<<<nblk, RS_THREADS, 0, st>>>(kin, vin, kout, vout, nkeys, shift, hist, nblk, total);
    PC_LAUNCH_CHECK();
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  k_bin_offsets<<<ceil_div((int64_t)nbins + 1, 256), 256, 0, st>>>(kin, nkeys, nbins, off);
  PC_LAUNCH_CHECK();
  const int* hoff = static_cast<const int*>(up.block(sizeof(int) * ((size_t)nbins + 1)));
  if (!hoff) return fail(PC_ERR_OOM, "plan: pinned memory for %u bins", nbins);
  PC_CUDA(cudaMemcpyAsync(const_cast<int*>(hoff), off, sizeof(int) * ((size_t)nbins + 1), cudaMemcpyDeviceToHost, st));
  PC_CUDA(cudaStreamSynchronize(st));
  p->n_slots = hoff[nbins];

  PC_TRY(dev_alloc_t(p, &p->slot_vis, (size_t)std::max<int64_t>(p->n_slots, 1)));
  PC_TRY(dev_alloc_t(p, &p->slot_geom, (size_t)std::max<int64_t>(p->n_slots, 1)));
  if (p->n_slots > 0) {
    k_slot_gather<<<ceil_div(p->n_slots, 256), 256, 0, st>>>(uvw, vin, p->n_slots, bg,
                                                             p->slot_vis, p->slot_geom);
    PC_LAUNCH_CHECK();
  }

  // ---- gridding sub-problems: the slot range of each (tile, plane group),
  // split into equal pieces of at most kMaxSlotsPerSub slots (multiples of 64,
  // the tensor-core stage) sized so that the pieces fill the GPU in about two
  // even waves of two CTAs per SM -- a few long sub-problems left over for a
  // second wave would otherwise double the gridding time.
  const int kMaxSlotsPerSub = 512;   // the autotuner's usual pick (smaller pieces: more CTAs in flight)
  // the slot range of each (tile, group of Q planes) that holds any; returns the slots
  auto plane_groups = [&](int Q, std::vector<int4>& out) {
    int64_t total = 0;
    for (int t = 0; t < p->nT * p->nT; ++t) {
      for (int gq = 0; gq < ceil_div(p->P, Q); ++gq) {
        int q0 = gq * Q;
        // plane starts whose footprint meets the group, widened to whole pairs
        // (the extra slots' footprints miss the group: zero weights there)
        int ps_lo = 0, ps_hi = 0;
        if (p->wstack) {
          ps_lo = std::max(0, q0 - p->W + 1);
          ps_hi = std::min(p->P - p->W, q0 + Q - 1);
        }
        if (ps_hi < ps_lo) continue;
        int s0 = hoff[(size_t)t * p->Pw + (ps_lo >> 1)];
        int s1 = hoff[(size_t)t * p->Pw + (ps_hi >> 1) + 1];
        if (s1 > s0) {
          out.push_back(make_int4(t, gq, s0, s1));
          total += s1 - s0;
        }
      }
    }
    return total;
  };
  std::vector<int4> ranges;
  const int64_t total_slots = plane_groups(p->Qg, ranges);
  int n_sm = 152;
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, p->device);
  const int64_t want = 4ll * n_sm;
  // without w-stacking the CUDA cores grid, and a CTA's time is its slots one after
  // the other: down to 32
  const int piece_min = p->wstack ? 128 : 32, stage = p->wstack ? 64 : 32;
  int piece = (int)std::min<int64_t>(kMaxSlotsPerSub, std::max<int64_t>(piece_min, (total_slots + want - 1) / want));
  piece = ceil_div(piece, stage) * stage;
  p->sub_ranges = ranges;
  // tile rows / columns that hold visibilities (the one-warp FFTs skip the rest, which stay zero)
  p->row_mask = p->col_mask = 0;
  if (p->nT <= 32)
    for (const int4& s : ranges) {
      p->row_mask |= 1u << (s.x / p->nT);
      p->col_mask |= 1u << (s.x % p->nT);
    }
  // room for the finest split: pieces of 32 or (the autotuner's) 64 slots
  p->sub_cap = (int)(total_slots / stage + (int64_t)ranges.size() + 1);
  PC_TRY(dev_alloc_t(p, &p->subs, (size_t)p->sub_cap));
  PC_TRY(split_subs(p, piece, up));
  // degridding over plane groups: its own groups and pieces. Its time is a thread's slots
  // one after the other, Qd planes each, and eight planes of a tile leave room for three
  // CTAs an SM: half the planes, or four beyond twelve. Pieces of whole passes of its 256
  // threads (in the gridding's 320 the second pass was nearly empty), 512 slots where
  // they still make five CTAs an SM. us, the gridding's groups and pieces and these: 512 x
  // 512, 200k visibilities, 8 planes 60 and 49, 11 planes 55 and 55, 15 planes 64 and 56;
  // 306 x 306, 118k, 8 planes 47 and 38; 400 x 400, 60k, 8 planes 35 and 29
  if (!grid_win_mode(p) || p->want_tune) {
    std::vector<int4> dr, ds;
    p->Qd = !p->wstack ? 1 : p->P <= 12 ? ceil_div(p->P, 2) : 4;
    const int64_t share = (plane_groups(p->Qd, dr) + want - 1) / want;
    const int dpiece = share >= 3 * 256 ? 512 : share > 192 ? 256 : share > 128 ? 192 : 128;
    for (const int4& r : dr) {
      const int n = ceil_div(r.w - r.z, dpiece), sz = ceil_div(r.w - r.z, n);
      for (int a = r.z; a < r.w; a += sz) ds.push_back(make_int4(r.x, r.y, a, std::min(r.w, a + sz)));
    }
    p->n_dsub = (int)ds.size();
    PC_TRY(dev_alloc_t(p, &p->dsubs, std::max<size_t>(ds.size(), 1)));
    PC_TRY(up.upload(p->dsubs, ds.data(), sizeof(int4) * ds.size()));
  }
  // window gridding: the bin offsets on the device, the tiles that hold slots,
  // and the CTA list (gwin::part_slots)
  PC_TRY(dev_alloc_t(p, &p->win_off, (size_t)nbins + 1));
  PC_CUDA(cudaMemcpyAsync(p->win_off, off, sizeof(int) * ((size_t)nbins + 1), cudaMemcpyDeviceToDevice, st));
  p->win_tiles.clear();
  for (int t = 0; t < p->nT * p->nT; ++t) {
    const int n = hoff[(size_t)(t + 1) * p->Pw] - hoff[(size_t)t * p->Pw];
    if (n > 0) p->win_tiles.push_back(make_int2(t, n));
  }
  p->wsub_cap = p->n_slots / 64 + (int64_t)p->win_tiles.size() + 1;
  PC_TRY(dev_alloc_t(p, &p->wsubs, (size_t)p->wsub_cap));
  const int n_tiles = (int)p->win_tiles.size();
  PC_TRY(split_wsubs(p, gwin::part_slots(p->n_slots, n_tiles, p->P, n_sm, 65536), up));
  PC_TRY(dev_alloc_t(p, &p->dwsubs, (size_t)p->wsub_cap));
  // window degridding: no part writes the grid, so 8192 also with many tiles (measured
  // best or within 2 % of the best on 2048^2 / 2M and 4096^2 / 10M; the tuner times it)
  PC_TRY(split_dwsubs(p, gwin::part_slots(p->n_slots, n_tiles, p->P, n_sm, 8192), up));
  // grid rows that any visibility can reach: the rows of tile rows with a sub-problem
  {
    std::vector<char> row_on(p->nT, 0);
    for (const int4& s : ranges) row_on[s.x / p->nT] = 1;
    std::vector<int> rows;
    for (int tv = 0; tv < p->nT; ++tv)
      if (row_on[tv])
        for (int b = 0; b < p->T; ++b) rows.push_back(tv * p->T + b);
    p->n_active_rows = (int)rows.size();
    PC_TRY(dev_alloc_t(p, &p->active_rows, std::max<size_t>(rows.size(), 1)));
    PC_TRY(up.upload(p->active_rows, rows.data(), sizeof(int) * rows.size()));
    // compact position of every grid row, and the column groups that can hold data
    std::vector<int> pos(p->G, -1);
    for (size_t c = 0; c < rows.size(); ++c) pos[rows[c]] = (int)c;
    PC_TRY(dev_alloc_t(p, &p->row_pos, (size_t)p->G));
    PC_TRY(up.upload(p->row_pos, pos.data(), sizeof(int) * p->G));
    std::vector<uint32_t> colw((size_t)std::max(1, p->G / 1024), 0u);
    for (const int4& s : ranges) {
      const int g = s.x % p->nT;                  // a tile column is one 32-column group
      colw[(size_t)g >> 5] |= 1u << (g & 31);
    }
    p->n_active_col_groups = 0;
    for (uint32_t word : colw) p->n_active_col_groups += __builtin_popcount(word);
    PC_TRY(dev_alloc_t(p, &p->col_bits, colw.size()));
    PC_TRY(up.upload(p->col_bits, colw.data(), sizeof(uint32_t) * colw.size()));
    if (fft_big_size(p->G)) {
      // the one-CTA passes' compact rows, allocated here (never inside a captured solve)
      const size_t nb = (size_t)ceil_div(std::max(p->n_active_rows, 1), 4);
      PC_TRY(p->xc.ensure(sizeof(float2) * (size_t)p->P * nb * Nt * 4));
      PC_TRY(make_xc_tensor_map(p));
    }
  }
  PC_CUDA(cudaStreamSynchronize(st));
  return PC_OK;
}

// Device bytes a plan and its solve may hold (an upper estimate used to admit
// jobs by memory): the gridding planes, the pass-1 FFT buffer, the pixel
// tables, the binned visibilities, the working set of the solver and the
// tensor-core phase buffer (chunked at 2 GB).
int64_t plan_bytes_estimate(int64_t M, int N, double fov, double w_min, double w_max, int W) {
  int64_t G = 32;
  while (G < 2 * N) G *= 2;
  const double dl = fov / N;
  const double half = 0.5 * N * dl;
  const double r2c = 2.0 * half * half;
  const double s_min = -r2c / (1.0 + std::sqrt(std::max(1.0 - r2c, 1e-12)));
  int64_t P = 1;
  if (M > 0 && w_max > w_min) {
    const double dw = 1.0 / (2.0 * (0.0 - s_min));
    P = (int64_t)std::ceil((w_max - w_min) / dw) + W;
  }
  const int64_t groups = (P + 7) / 8;
  const int64_t NN = (int64_t)N * N;
  int64_t b = 0;
  b += P * G * G * 8;                       // grid planes
  b += P * N * G * 8;                       // pass-1 FFT output
  b += NN * (16 + 16 + 4 + 1 + 4);          // pixel and atom tables, mu, marks, selection
  b += M * (16 + 8);                        // fixed-point visibilities, residual
  b += M * groups * 2 * 24;                 // binned slots (replication into tiles and plane groups)
  b += 2 * 4096ll * 4096ll * 4;             // Gram working set (grown on demand; 4096 atoms)
  b += std::min<int64_t>(2ll << 30, 1024 * M * 8);   // phase buffer of the tensor-core Gram
  b += 64ll << 20;                          // scratch
  return b;
}

}  // namespace pc

using namespace pc;

extern "C" int pc_plan_create(const double* uvw_dev, int64_t M, int32_t N, double fov_rad,
                              const pc_plan_opts* opts, void* stream, pc_plan_t* plan_out) {
  clear_error();
  if (!plan_out) return fail(PC_ERR_INVALID_ARG, "pc_plan_create: plan_out is NULL");
  *plan_out = nullptr;
  if (opts && opts->version != PC_ABI_VERSION)
    return fail(PC_ERR_INVALID_ARG, "pc_plan_create: opts->version %d != %d", opts->version,
                PC_ABI_VERSION);
  if (M < 0 || M > (1ll << 29))
    return fail(PC_ERR_INVALID_ARG, "pc_plan_create: M = %lld out of range [0, 2^29]", (long long)M);
  if (N < 16 || N > 4096 || (N & 1))
    return fail(PC_ERR_INVALID_ARG, "pc_plan_create: N = %d must be even and in [16, 4096]", N);
  if (!(fov_rad > 0.0) || !(fov_rad < 1.4))
    return fail(PC_ERR_INVALID_ARG, "pc_plan_create: fov_rad = %g must be in (0, 1.4)", fov_rad);
  if (M > 0 && !is_device_ptr(uvw_dev))
    return fail(PC_ERR_INVALID_ARG, "pc_plan_create: uvw_dev is not a device pointer");
  int W = (opts && opts->kernel_width) ? opts->kernel_width : 7;
  int T = (opts && opts->tile) ? opts->tile : 32;
  int maxP = (opts && opts->max_planes) ? opts->max_planes : 256;
  if (W < 4 || W > kMaxW) return fail(PC_ERR_INVALID_ARG, "pc_plan_create: kernel_width %d not in [4, 8]", W);
  if (T != 32) return fail(PC_ERR_INVALID_ARG, "pc_plan_create: tile %d must be 32", T);
  if (maxP < 1 || maxP > 4096) return fail(PC_ERR_INVALID_ARG, "pc_plan_create: max_planes %d", maxP);
  const int grid_mode = opts ? opts->grid_mode : 0;
  if (grid_mode < 0 || grid_mode > 3)
    return fail(PC_ERR_INVALID_ARG, "pc_plan_create: grid_mode %d not in [0, 3]", grid_mode);
  const int tune = opts ? opts->autotune : 0;
  if (tune != 0 && tune != 1) return fail(PC_ERR_INVALID_ARG, "pc_plan_create: autotune must be 0 or 1");
  const int fft_kernel = opts ? opts->fft_kernel : 0;
  if (fft_kernel != 0 && fft_kernel != 1)
    return fail(PC_ERR_INVALID_ARG, "pc_plan_create: fft_kernel must be 0 or 1");

  pc_plan_s* p = new pc_plan_s();
  cudaGetDevice(&p->device);
  p->M = M;
  p->N = N;
  p->fov = fov_rad;
  p->W = W;
  p->T = T;
  p->grid_mode = grid_mode;
  p->fft_warp = fft_kernel == 1 ? 0 : -1;
  p->want_tune = tune == 1;
  int rc = build_plan(p, uvw_dev, (cudaStream_t)stream, maxP);
  if (rc == PC_OK && tune) rc = autotune(p, (cudaStream_t)stream);
  if (rc != PC_OK) {
    pc_plan_destroy(p);
    return rc;
  }
  *plan_out = p;
  return PC_OK;
}

extern "C" int pc_plan_tuning_info(pc_plan_t p, pc_plan_tuning* out) {
  clear_error();
  if (!p || !out) return fail(PC_ERR_INVALID_ARG, "pc_plan_tuning_info: NULL argument");
  out->tuned = p->tuned ? 1 : 0;
  out->grid_mode = grid_win_mode(p) ? 3 : (p->wstack && p->grid_mode != 1) ? 2 : 1;
  out->grid_piece = grid_win_mode(p) ? p->win_cap : p->grid_piece;
  int R = p->fft_R > 0 ? p->fft_R : fft_rows_per_cta(p);
  const bool rw = fft_rows_warp(p) || fft_rows_big(p), cw = fft_cols_warp(p) || fft_cols_big(p);
  out->fft_rows_per_cta = fft_rows_big(p) ? 1 : rw ? 8 : std::min(std::max(R, 1), 32);
  out->grid_us = p->tune_grid_us;
  out->fft_rows_us = p->tune_fft_us;
  out->fft_cols_planes = cw ? 1 : cols_planes_per_pass(p);
  out->fft_cols_us = p->tune_fft_cols_us;
  out->fft_warp = (rw ? 1 : 0) | (cw ? 2 : 0);
  out->degrid_piece = grid_win_mode(p) ? p->dwin_cap : 0;
  out->reserved = 0;
  out->degrid_us = p->tune_degrid_us;
  return PC_OK;
}

extern "C" void pc_plan_destroy(pc_plan_t p) {
  if (!p) return;
  // the buffers may still be in use on any stream: wait for the device once
  // (as cudaFree would), then return them to the pool
  cudaDeviceSynchronize();
  for (void* q : p->owned) dfree(q, 0);
  if (p->readback) pinned_put(p->readback);
  if (p->atoms_read) cudaEventDestroy(p->atoms_read);
  p->atomsA.release();
  p->atomsB.release();
  p->idxA.release();
  p->idxB.release();
  p->xA.release();
  p->xB.release();
  p->oldpos.release();
  p->newrows.release();
  p->keep.release();
  p->GA.release();
  p->GB.release();
  p->bA.release();
  p->bB.release();
  p->acc.release();
  p->perm.release();
  p->atomsP.release();
  p->pbuf.release();
  p->degrid_buf.release();
  p->xc.release();
  p->opw.release();
  p->dirty.release();
  if (p->dict) {
    p->dict->release();
    delete p->dict;
  }
  if (p->scache) {
    p->scache->release();
    delete p->scache;
  }
  delete p;
}

extern "C" int pc_plan_reach(pc_plan_t p, int32_t* rows, int32_t* col_groups) {
  clear_error();
  if (!p) return fail(PC_ERR_INVALID_ARG, "pc_plan_reach: NULL plan");
  if (rows) *rows = p->n_active_rows;
  if (col_groups) *col_groups = p->n_active_col_groups;
  return PC_OK;
}

extern "C" int pc_plan_transforms(pc_plan_t p, int32_t* grid_side, int32_t* image_side) {
  clear_error();
  if (!p) return fail(PC_ERR_INVALID_ARG, "pc_plan_transforms: NULL plan");
  if (grid_side) *grid_side = p->G;
  if (image_side) *image_side = p->Nt;
  return PC_OK;
}

extern "C" int pc_plan(const double* uvw_dev, int64_t M, int32_t N, double fov_rad,
                       const pc_plan_opts* opts, void* stream, pc_plan_t* plan_out) {
  return pc_plan_create(uvw_dev, M, N, fov_rad, opts, stream, plan_out);
}

extern "C" int pc_plan_info(pc_plan_t p, int32_t* grid_side, int32_t* tile, int32_t* n_planes,
                            int64_t* n_slots, int32_t* kernel_width, double* dw) {
  if (!p) return fail(PC_ERR_INVALID_ARG, "pc_plan_info: NULL plan");
  if (grid_side) *grid_side = p->G_image;
  if (tile) *tile = p->T;
  if (n_planes) *n_planes = p->P;
  if (n_slots) *n_slots = p->n_slots;
  if (kernel_width) *kernel_width = p->W;
  if (dw) *dw = p->dw;
  return PC_OK;
}
