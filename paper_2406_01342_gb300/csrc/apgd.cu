// Restricted LASSO solve of step 2 of Algorithm 2 by accelerated proximal
// gradient (FISTA, the APGD the paper names in Sect. 4.4 / 4.1) on the Gram
// form of the support problem:
//
//   f(x) = 1/2 x^T G x - b^T x + lambda ||x||_1,   G = Re(Phi_S^H Phi_S), b = Re(Phi_S^H V)
//
// Readings (the paper gives no constants): step 1/L with L = 1.01 x the
// largest eigenvalue of G; the monotone FISTA variant; stop when
// ||z - y|| <= eps ||z||. The eigenvalue comes from Lanczos on G started from
// the all-ones vector: the largest Ritz value of the tridiagonal matrix (by
// Sturm-count multisection), until it changes by < 1e-5 relative between
// checks every 4 steps, at most 64 steps (or n, or an invariant subspace).
// Ritz values approach the top eigenvalue from below and converge faster than
// linearly, so the 1 % margin of L covers the remaining error many times.
//
// GB300 mapping: one CTA up to 224 atoms (k_apgd_cta), a thread-block cluster of
// 8 or 16 beyond (k_apgd_full), one CTA per SM where a cluster cannot hold G
// (k_apgd_grid), and k_apgd where the full vectors do not fit: a cluster whose CTA r
// owns a contiguous block of rows of G and of every vector. Each of its iterations
// does one GEMV: the CTAs publish their slice of the proximal point z in shared
// memory, a cluster barrier, every CTA gathers the whole z through distributed
// shared memory, multiplies its rows, publishes its partial sums, a second
// barrier, and every CTA reduces the partials in the same order (so all take
// identical decisions). G z is the only matrix product per iteration: G y and
// G x are kept as linear combinations of previous products.
//
// Arithmetic: FP32 vectors and no float64 instruction in any loop (float64 has
// a low rate and long dependent latency on this GPU; it made an iteration take
// ~10 us). The monotone test F(z) <= F(x) needs the sign of a difference of two
// ~1e7 numbers: the full-vector kernel sums the difference directly as
// sum_i (z_i - x_i)((Gz_i + Gx_i)/2 - b_i) + lambda(|z_i| - |x_i|), whose terms
// all vanish as z -> x, in FP32; the row-slice kernel (large supports) carries
// the objective itself as double-float pairs (hi + lo, exact products and
// error-free sums, ~44 bits).
#include <cooperative_groups.h>

#include <cmath>

#include "apgd_rows.cuh"
#include "lanczos.cuh"
#include "pc_internal.cuh"

namespace cg = cooperative_groups;

namespace pc {
namespace {

// ---- double-float arithmetic (Dekker / Knuth error-free transformations)
struct Df {
  float hi, lo;
};

__device__ __forceinline__ Df df_two_sum(float a, float b) {
  const float s = a + b;
  const float bb = s - a;
  const float e = (a - (s - bb)) + (b - bb);
  return {s, e};
}
__device__ __forceinline__ Df df_add(Df a, Df b) {
  Df s = df_two_sum(a.hi, b.hi);
  const float e = s.lo + a.lo + b.lo;
  const float hi = s.hi + e;
  return {hi, e - (hi - s.hi)};
}
__device__ __forceinline__ Df df_prod(float a, float b) {   // exact a * b
  const float p = a * b;
  return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ Df df_scale(Df a, float b) {
  const float p = a.hi * b;
  float e = fmaf(a.hi, b, -p);
  e = fmaf(a.lo, b, e);
  const float hi = p + e;
  return {hi, e - (hi - p)};
}
__device__ __forceinline__ Df df_neg(Df a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ bool df_le(Df a, Df b) {          // a <= b
  const Df d = df_add(a, df_neg(b));
  return d.hi < 0.f || (d.hi == 0.f && d.lo <= 0.f);
}
__device__ __forceinline__ Df df_shfl_xor(Df a, int off) {
  return {__shfl_xor_sync(0xffffffffu, a.hi, off), __shfl_xor_sync(0xffffffffu, a.lo, off)};
}

struct ApgdArgs {
  const float* G;
  int ldg;
  const float* b;
  int n;
  float lam;
  float eps;
  int max_iter;
  float* x;
  int* out_iters;
  double* out_L;
  double* out_F;
  int* out_lanczos;
  int* err;       // set to 1 if a bounded wait expired (may be null)
  int positive;   // 1: x >= 0 (proximal map max(z - lambda/L, 0))
  int rows_per;
  int n_pad;
  int cache;      // rows of G that a CTA keeps in shared memory (k_apgd: 1 for all, 0 for none)
  int vec_ok;     // 1: float4 loads of G rows are aligned
  int scalar;     // a lane takes single columns, not groups of four
};

// Rows [r0, r0 + nr) of G (leading dimension ldg, n columns) into dst (row
// stride ld floats, ld a multiple of 4, dst 16-byte aligned), columns [n, ld)
// zero, by asynchronous copies: a warp per row, no register round trip per
// element, so every load of the block is in flight at once. The calling
// thread's copies are complete on return; the caller's barrier publishes them.
__device__ void load_rows_async(float* dst, int ld, const float* __restrict__ G, int ldg, int r0, int nr,
                                int n, bool vec) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int r = warp; r < nr; r += nw) {
    const float* src = G + (size_t)(r0 + r) * ldg;
    float* d = dst + (size_t)r * ld;
    if (vec) {
      for (int c = 4 * lane; c < ld; c += 128) {
        const int bytes = max(0, min(16, (n - c) * 4));
        const uint32_t da = (uint32_t)__cvta_generic_to_shared(d + c);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(da), "l"(bytes > 0 ? src + c : src),
                     "r"(bytes)
                     : "memory");
      }
    } else {
      for (int c = lane; c < ld; c += 32) {
        if (c < n) {
          const uint32_t da = (uint32_t)__cvta_generic_to_shared(d + c);
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(da), "l"(src + c) : "memory");
        } else {
          d[c] = 0.f;
        }
      }
    }
  }
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// Several independent restricted problems in one launch: cluster c of the
// grid solves job c (all jobs of a launch share the cluster size).
constexpr int APGD_BATCH_MAX = 16;
struct ApgdBatch {
  ApgdArgs job[APGD_BATCH_MAX];
  int n_jobs;
};

constexpr int APGD_THREADS = 256;
constexpr int NPART = 5;

struct Smem {
  float* zfull;   // n_pad
  float* pub;     // rows_per (published slice)
  float* y;
  float* Gy;
  float* x;
  float* Gx;
  float* z;
  float* Gz;
  float* bb;
  Df* part;       // 2 buffers of 8 partial sums (the second for back-to-back reductions)
  float* Gc;      // rows_per * n_pad (optional)
};

__device__ Smem carve(float* base, const ApgdArgs& a) {
  Smem s;
  float* p = base;
  s.zfull = p; p += a.n_pad;
  s.pub = p; p += a.rows_per;
  s.y = p; p += a.rows_per;
  s.Gy = p; p += a.rows_per;
  s.x = p; p += a.rows_per;
  s.Gx = p; p += a.rows_per;
  s.z = p; p += a.rows_per;
  s.Gz = p; p += a.rows_per;
  s.bb = p; p += a.rows_per;
  p = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(p) + 15) & ~uintptr_t(15));
  s.part = reinterpret_cast<Df*>(p); p += 2 * 16;
  s.Gc = p;
  return s;
}

// Gather the published slices of every CTA into zfull.
__device__ void gather(cg::cluster_group& cl, const Smem& s, const ApgdArgs& a) {
  for (int idx = threadIdx.x; idx < a.n; idx += blockDim.x) {
    const int rr = idx / a.rows_per;
    const int off = idx - rr * a.rows_per;
    const float* remote = cl.map_shared_rank(s.pub, rr);
    s.zfull[idx] = remote[off];
  }
  for (int idx = a.n + threadIdx.x; idx < a.n_pad; idx += blockDim.x) s.zfull[idx] = 0.f;
}

// out[r] = G[r0 + r, :] . zfull for the nr own rows. A warp takes 4 rows at
// a time (independent accumulators and shuffle chains, so their latencies
// overlap); full float4 groups inside [0, n), then a scalar tail: columns >= n
// of a caller's G are never read.
__device__ void gemv_rows(const Smem& s, const ApgdArgs& a, int r0, int nr, float* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const bool vec = a.cache || a.vec_ok;
  const int n4 = a.n >> 2;
  const float4* z4 = reinterpret_cast<const float4*>(s.zfull);
  for (int rb = 4 * warp; rb < nr; rb += 4 * nw) {
    const float* rows[4];
    float acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = min(rb + q, nr - 1);
      rows[q] = a.cache ? s.Gc + (size_t)r * a.n_pad : a.G + (size_t)(r0 + r) * a.ldg;
      acc[q] = 0.f;
    }
    if (vec) {
      for (int c = lane; c < n4; c += 32) {
        const float4 z = z4[c];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 g = reinterpret_cast<const float4*>(rows[q])[c];
          acc[q] = fmaf(g.x, z.x, acc[q]);
          acc[q] = fmaf(g.y, z.y, acc[q]);
          acc[q] = fmaf(g.z, z.z, acc[q]);
          acc[q] = fmaf(g.w, z.w, acc[q]);
        }
      }
      for (int c = 4 * n4 + lane; c < a.n; c += 32)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = fmaf(rows[q][c], s.zfull[c], acc[q]);
    } else {
      for (int c = lane; c < a.n; c += 32)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = fmaf(rows[q][c], s.zfull[c], acc[q]);
    }
    for (int off = 16; off; off >>= 1)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
    if (lane < 4 && rb + lane < nr) {
      float v = acc[0];
#pragma unroll
      for (int q = 1; q < 4; ++q)
        if (lane == q) v = acc[q];
      out[rb + lane] = v;
    }
  }
}

// Double-float sums of NPART values over the block's first APGD_THREADS threads, written to part[].
__device__ void block_sums(Df v[NPART], Df* part, Df* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = APGD_THREADS / 32;
  for (int off = 16; off; off >>= 1)
#pragma unroll
    for (int q = 0; q < NPART; ++q) v[q] = df_add(v[q], df_shfl_xor(v[q], off));
  if (lane == 0 && warp < nw)
#pragma unroll
    for (int q = 0; q < NPART; ++q) scratch[warp * NPART + q] = v[q];
  __syncthreads();
  if (warp == 0) {   // the nw (<= 8) warp sums: a 3-level butterfly in warp 0
#pragma unroll
    for (int q = 0; q < NPART; ++q) v[q] = lane < nw ? scratch[lane * NPART + q] : Df{0.f, 0.f};
    for (int off = 4; off; off >>= 1)
#pragma unroll
      for (int q = 0; q < NPART; ++q) v[q] = df_add(v[q], df_shfl_xor(v[q], off));
    if (lane < NPART) {
      Df t = v[0];
#pragma unroll
      for (int q = 1; q < NPART; ++q)
        if (lane == q) t = v[q];
      part[lane] = t;
    }
  }
  __syncthreads();
}

// Sum the published partials of all CTAs: warp 0 reads each CTA's partials
// once over distributed shared memory and reduces them with a fixed butterfly
// (the same order in every CTA, so every CTA takes the same decisions).
__device__ void cluster_sums(cg::cluster_group& cl, Df* part, Df* s_tot, Df out[NPART]) {
  const int CS = (int)cl.num_blocks();
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const Df* rp = lane < CS ? cl.map_shared_rank(part, lane) : nullptr;
    Df v[NPART];
#pragma unroll
    for (int q = 0; q < NPART; ++q) v[q] = rp ? rp[q] : Df{0.f, 0.f};
    for (int off = 16; off; off >>= 1)
#pragma unroll
      for (int q = 0; q < NPART; ++q) v[q] = df_add(v[q], df_shfl_xor(v[q], off));
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < NPART; ++q) s_tot[q] = v[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < NPART; ++q) out[q] = s_tot[q];
}

__global__ void __launch_bounds__(APGD_THREADS, 1) k_apgd(const __grid_constant__ ApgdBatch batch) {
  extern __shared__ __align__(16) float apgd_sm[];
  __shared__ Df scratch[(APGD_THREADS / 32) * NPART];
  __shared__ Df s_tot[NPART];
  __shared__ float s_al[LZ_MAX], s_be[LZ_MAX], s_theta;
  cg::cluster_group cl = cg::this_cluster();
  const ApgdArgs& a = batch.job[blockIdx.x / cl.num_blocks()];
  const int rank = (int)cl.block_rank();
  const Smem s = carve(apgd_sm, a);
  const int r0 = rank * a.rows_per;
  const int nr = max(0, min(a.n, r0 + a.rows_per) - r0);
  Df* part2 = s.part + 8;

  if (a.cache) load_rows_async(s.Gc, a.n_pad, a.G, a.ldg, r0, nr, a.n, a.vec_ok != 0);
  const float v0 = rsqrtf((float)a.n);        // Lanczos start: all ones / sqrt(n)
  for (int r = threadIdx.x; r < a.rows_per; r += blockDim.x) {
    const bool own = r < nr;
    s.bb[r] = own ? a.b[r0 + r] : 0.f;
    s.x[r] = own ? a.x[r0 + r] : 0.f;
    s.y[r] = own ? v0 : 0.f;    // v_j
    s.z[r] = 0.f;               // v_{j-1}
    s.pub[r] = own ? v0 : 0.f;
  }
  __syncthreads();

  // ---- Lipschitz constant: Lanczos (alpha = v^T G v, then beta = ||w||)
  float theta = 0.f, theta_prev = 0.f, beta_prev = 0.f;
  int m = 0;
  for (int j = 0; j < LZ_MAX; ++j) {
    cl.sync();
    gather(cl, s, a);
    __syncthreads();
    gemv_rows(s, a, r0, nr, s.Gz);                  // w = G v_j
    __syncthreads();
    Df v[NPART] = {};
    for (int r = threadIdx.x; r < nr; r += blockDim.x) v[0] = df_add(v[0], df_prod(s.y[r], s.Gz[r]));
    block_sums(v, s.part, scratch);
    cl.sync();
    Df tot[NPART];
    cluster_sums(cl, s.part, s_tot, tot);
    const float alpha = tot[0].hi + tot[0].lo;
    Df v2[NPART] = {};
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
      const float w = s.Gz[r] - alpha * s.y[r] - beta_prev * s.z[r];
      s.Gz[r] = w;
      v2[0] = df_add(v2[0], df_prod(w, w));
    }
    block_sums(v2, part2, scratch);
    cl.sync();
    cluster_sums(cl, part2, s_tot, tot);
    const float beta = sqrtf(fmaxf(tot[0].hi + tot[0].lo, 0.f));
    if (threadIdx.x == 0) {
      s_al[j] = alpha;
      s_be[j] = beta;
    }
    m = j + 1;
    __syncthreads();
    const bool last = (m == a.n) || (m == LZ_MAX) || !(beta > 1e-7f * fabsf(alpha));
    if (last || (m % 4) == 0) {
      theta = tridiag_top(s_al, s_be, m, &s_theta);
      if (last || fabsf(theta - theta_prev) <= LZ_TOL * fabsf(theta)) break;
      theta_prev = theta;
    }
    const float inv = 1.f / beta;
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
      const float vn = s.Gz[r] * inv;
      s.z[r] = s.y[r];
      s.y[r] = vn;
      s.pub[r] = vn;
    }
    beta_prev = beta;
  }
  const float L = 1.01f * (theta > 0.f ? theta : 1.f);
  const float invL = 1.f / L;
  const float thr = a.lam * invL;

  // ---- initial G x
  for (int r = threadIdx.x; r < nr; r += blockDim.x) s.pub[r] = s.x[r];
  cl.sync();
  gather(cl, s, a);
  __syncthreads();
  gemv_rows(s, a, r0, nr, s.Gx);
  __syncthreads();
  Df Fx;
  {
    Df v[NPART] = {};
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
      v[0] = df_add(v[0], df_prod(s.x[r], s.Gx[r]));
      v[1] = df_add(v[1], df_prod(s.bb[r], s.x[r]));
      v[2] = df_add(v[2], Df{fabsf(s.x[r]), 0.f});
    }
    block_sums(v, s.part, scratch);
    cl.sync();
    Df tot[NPART];
    cluster_sums(cl, s.part, s_tot, tot);
    Fx = df_add(df_add(df_scale(tot[0], 0.5f), df_neg(tot[1])), df_scale(tot[2], a.lam));
  }
  for (int r = threadIdx.x; r < nr; r += blockDim.x) {
    s.y[r] = s.x[r];
    s.Gy[r] = s.Gx[r];
  }
  __syncthreads();

  // ---- monotone FISTA
  float t = 1.f;
  int it = 0;
  for (it = 1; it <= a.max_iter; ++it) {
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
      const float u = s.y[r] - (s.Gy[r] - s.bb[r]) * invL;
      const float zr = (a.positive ? fmaxf(u - thr, 0.f) : copysignf(fmaxf(fabsf(u) - thr, 0.f), u));
      s.z[r] = zr;
      s.pub[r] = zr;
    }
    cl.sync();
    gather(cl, s, a);
    __syncthreads();
    gemv_rows(s, a, r0, nr, s.Gz);
    __syncthreads();
    Df v[NPART] = {};
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
      const float zr = s.z[r];
      v[0] = df_add(v[0], df_prod(zr, s.Gz[r]));
      v[1] = df_add(v[1], df_prod(s.bb[r], zr));
      v[2] = df_add(v[2], Df{fabsf(zr), 0.f});
      const float d = zr - s.y[r];
      v[3] = df_add(v[3], df_prod(d, d));
      v[4] = df_add(v[4], df_prod(zr, zr));
    }
    block_sums(v, s.part, scratch);
    cl.sync();
    Df tot[NPART];
    cluster_sums(cl, s.part, s_tot, tot);
    const Df Fz = df_add(df_add(df_scale(tot[0], 0.5f), df_neg(tot[1])), df_scale(tot[2], a.lam));
    const float step = sqrtf(tot[3].hi + tot[3].lo);
    const float nz = sqrtf(tot[4].hi + tot[4].lo);
    const float t1 = 0.5f * (1.f + sqrtf(1.f + 4.f * t * t));
    const bool accept = df_le(Fz, Fx);
    const float c1 = t / t1, c2 = (t - 1.f) / t1;
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
      const float xo = s.x[r], Gxo = s.Gx[r];
      const float xn = accept ? s.z[r] : xo;
      const float Gxn = accept ? s.Gz[r] : Gxo;
      s.y[r] = xn + c1 * (s.z[r] - xn) + c2 * (xn - xo);
      s.Gy[r] = Gxn + c1 * (s.Gz[r] - Gxn) + c2 * (Gxn - Gxo);
      s.x[r] = xn;
      s.Gx[r] = Gxn;
    }
    if (accept) Fx = Fz;
    t = t1;
    __syncthreads();
    if (step <= a.eps * nz) break;
  }
  if (it > a.max_iter) it = a.max_iter;
  for (int r = threadIdx.x; r < nr; r += blockDim.x) a.x[r0 + r] = s.x[r];
  if (rank == 0 && threadIdx.x == 0) {
    if (a.out_iters) *a.out_iters = it;
    if (a.out_L) *a.out_L = (double)L;
    if (a.out_F) *a.out_F = (double)Fx.hi + (double)Fx.lo;
    if (a.out_lanczos) *a.out_lanczos = m;
  }
  cl.sync();   // no CTA leaves while others may still read its shared memory
}

// FP32 sums of K values over the block's first APGD_THREADS threads (a fixed
// butterfly: the same inputs give the same sums in every CTA), for every thread. One
// barrier: the buffers alternate, and every thread adds the eight warps' sums.
template <int K>
__device__ __forceinline__ void block_sum_f(float (&v)[K], float (*red)[3][8], int& parity) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < APGD_THREADS / 32) {
    for (int off = 16; off; off >>= 1)
#pragma unroll
      for (int q = 0; q < K; ++q) v[q] += __shfl_xor_sync(0xffffffffu, v[q], off);
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < K; ++q) red[parity][q][warp] = v[q];
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < K; ++q) {
    const float4 f = *reinterpret_cast<const float4*>(&red[parity][q][0]);
    const float4 h = *reinterpret_cast<const float4*>(&red[parity][q][4]);
    v[q] = ((f.x + h.x) + (f.z + h.z)) + ((f.y + h.y) + (f.w + h.w));
  }
  parity ^= 1;
}

// ---------------------------------------------------------------------------
// Full-vector variant (used whenever its vectors fit): every CTA keeps all n
// entries of x, y, z, Gx, Gy and b, and owns rows [r0, r0 + nr) of G (nr a
// multiple of 4 except in the last CTA), as many of them in shared memory as fit;
// the others are read from L2 each time, 16 loads of 16 bytes in flight a thread.
// A warp multiplies four rows by the (local) full vector and sends the four sums
// to every CTA of the cluster, a lane to each, as one asynchronous 16-byte store
// whose bytes complete on the receiver's mbarrier; every thread then waits
// (bounded) on its CTA's mbarrier until all entries have landed. No cluster
// barrier and no remote loads sit on the iteration path, only the one-way
// latency of the stores. The reductions and updates are then done redundantly
// over all n entries -- identical data and order in every CTA, hence identical
// decisions. Every thread keeps to its own entries of the vectors, so that an
// iteration crosses two block barriers (input vector complete; partial sums
// complete).
//
// Two receive buffers alternate. A CTA sends product i + 2 into buffer i mod 2
// only after it has received every CTA's product i + 1, which each CTA (all have
// rows, see cluster_slice) sends only after it has consumed product i, so a buffer is
// never overwritten while it is read. The mbarrier of a buffer is re-armed for product i + 2 before this CTA
// sends product i + 1, and no phase can end twice while a thread still waits for
// its first end: product i + 2 needs this CTA's own rows, which it sends after a
// barrier of all its threads.
//
// What bounds it: up to 800 atoms the latency of exchange, barriers and sums;
// beyond, the rows that 16 SMs cannot keep, read from L2. Measured against bulk
// copies of slices with six barriers an iteration, all rows or none in shared
// memory, us an iteration before and after: 300 atoms 2.30 and 1.56, 500 2.46 and
// 1.79, 900 5.5 and 3.8, 1300 7.2 and 5.7, 2500 16.8 and 16.0.

constexpr long long APGD_WAIT_CYCLES = 4000000000ll;   // ~2 s at 2 GHz

struct SmemF {
  float* rx0;     // n_pad each: the two receive buffers of the products
  float* rx1;
  float* x;       // n_pad each, full vectors
  float* Gx;
  float* y;
  float* Gy;
  float* z;
  float* bb;
  float* Gc;      // cache x n_pad
};

__device__ SmemF carve_full(float* base, const ApgdArgs& a) {
  SmemF s;
  float* p = base;
  s.rx0 = p; p += a.n_pad;
  s.rx1 = p; p += a.n_pad;
  s.x = p; p += a.n_pad;
  s.Gx = p; p += a.n_pad;
  s.y = p; p += a.n_pad;
  s.Gy = p; p += a.n_pad;
  s.z = p; p += a.n_pad;
  s.bb = p; p += a.n_pad;
  s.Gc = p;
  return s;
}

__device__ __forceinline__ uint32_t cluster_addr(uint32_t saddr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arm(uint32_t mbar, uint32_t tx) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(tx) : "memory");
}
__device__ __forceinline__ bool mbar_try_cluster(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(mbar), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ bool mbar_wait_cluster(uint32_t mbar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try_cluster(mbar, parity))
    if (clock64() - t0 > APGD_WAIT_CYCLES) return false;
  return true;
}

struct Exchange {
  uint32_t rx0, rx1;     // shared::cta addresses of the receive buffers
  uint32_t bar0, bar1;   // ... and of their mbarriers
  uint32_t phase;        // parity bit per buffer
  int buf;
  int CS;
  __device__ uint32_t rx(int b) const { return b ? rx1 : rx0; }
  __device__ uint32_t bar(int b) const { return b ? bar1 : bar0; }
};

// Four rows of G by a vector in shared memory: the lane's part. U: steps of the
// column loop whose loads are issued together.
template <int U>
__device__ __forceinline__ void rows_dot(const float* const (&rows)[4], const float* vec, int n, bool vecld,
                                         float (&acc)[4]) {
  const int lane = threadIdx.x & 31, n4 = n >> 2;
  const float4* v4 = reinterpret_cast<const float4*>(vec);
  if (vecld) {
#pragma unroll U
    for (int c = lane; c < n4; c += 32) {
      const float4 z = v4[c];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 g = reinterpret_cast<const float4*>(rows[q])[c];
        acc[q] = fmaf(g.x, z.x, acc[q]);
        acc[q] = fmaf(g.y, z.y, acc[q]);
        acc[q] = fmaf(g.z, z.z, acc[q]);
        acc[q] = fmaf(g.w, z.w, acc[q]);
      }
    }
    for (int c = 4 * n4 + lane; c < n; c += 32)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fmaf(rows[q][c], vec[c], acc[q]);
  } else {
#pragma unroll U
    for (int c = lane; c < n; c += 32)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fmaf(rows[q][c], vec[c], acc[q]);
  }
}

// G vec for all n rows, in every CTA; returns the receive buffer holding it.
// *bad is set if the bounded wait expired: read it behind the next barrier. The
// caller's barriers order the vector's writes before and its next ones after.
__device__ float* cluster_gemv(const ApgdArgs& a, const SmemF& s, const float* vec, int r0, int nr,
                               Exchange& ex, int* bad) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int b = ex.buf;
  // rows from L2 first, the cached ones after
  const int n_groups = (nr + 3) >> 2;
  for (int gi = n_groups - 1 - warp; gi >= 0; gi -= nw) {
    const int rb = 4 * gi;
    const float* rows[4];
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    if (rb < a.cache) {                               // cache: a multiple of 4, or at least nr
#pragma unroll
      for (int q = 0; q < 4; ++q) rows[q] = s.Gc + (size_t)min(rb + q, nr - 1) * a.n_pad;
      rows_dot<2>(rows, vec, a.n, !a.scalar, acc);
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) rows[q] = a.G + (size_t)(r0 + min(rb + q, nr - 1)) * a.ldg;
      rows_dot<4>(rows, vec, a.n, a.vec_ok != 0, acc);
    }
    for (int off = 16; off; off >>= 1)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
    if (lane < ex.CS) {
#pragma unroll
      for (int q = 1; q < 4; ++q)
        if (rb + q >= nr) acc[q] = 0.f;               // past the last row: fills the vectors' padding
      asm volatile(
          "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
              cluster_addr(ex.rx(b) + (uint32_t)(r0 + rb) * 4u, lane)),
          "r"(__float_as_uint(acc[0])), "r"(__float_as_uint(acc[1])), "r"(__float_as_uint(acc[2])),
          "r"(__float_as_uint(acc[3])), "r"(cluster_addr(ex.bar(b), lane))
          : "memory");
    }
  }
  if (!mbar_wait_cluster(ex.bar(b), (ex.phase >> b) & 1u)) *bad = 1;
  ex.phase ^= 1u << b;
  ex.buf ^= 1;
  // re-arm for this buffer's next use (two products from now)
  if (threadIdx.x == 0) mbar_arm(ex.bar(b), (uint32_t)a.n_pad * 4u);
  return b ? s.rx1 : s.rx0;
}

template <int THREADS>   // the first APGD_THREADS hold the vectors, all of them multiply
__global__ void __launch_bounds__(THREADS, 1) k_apgd_full(const __grid_constant__ ApgdBatch batch) {
  extern __shared__ __align__(16) float apgdf_sm[];
  __shared__ Df scratch[(APGD_THREADS / 32) * NPART];
  __shared__ Df s_part[NPART];
  __shared__ __align__(16) float s_red[2][3][8];
  __shared__ int s_bad;
  __shared__ float s_al[LZ_MAX], s_be[LZ_MAX], s_theta;
  __shared__ __align__(8) uint64_t s_rxbar[2];
  cg::cluster_group cl = cg::this_cluster();
  const ApgdArgs& a = batch.job[blockIdx.x / cl.num_blocks()];
  const int rank = (int)cl.block_rank();
  const SmemF s = carve_full(apgdf_sm, a);
  const RowSlice own = cluster_slice(a.n, (int)cl.num_blocks(), rank);
  const int r0 = own.r0, nr = own.nr;
  const int n = a.n, tid = threadIdx.x, nt = APGD_THREADS;
  const int e0 = tid < nt ? tid : a.n_pad;    // first own entry of the vectors (none past the first threads)
  bool ok = true;
  int parity = 0;

  Exchange ex;
  ex.rx0 = (uint32_t)__cvta_generic_to_shared(s.rx0);
  ex.rx1 = (uint32_t)__cvta_generic_to_shared(s.rx1);
  ex.bar0 = (uint32_t)__cvta_generic_to_shared(&s_rxbar[0]);
  ex.bar1 = (uint32_t)__cvta_generic_to_shared(&s_rxbar[1]);
  ex.phase = 0;
  ex.buf = 0;
  ex.CS = (int)cl.num_blocks();
  if (tid == 0) {
    s_bad = 0;
    for (int b = 0; b < 2; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(ex.bar(b)));
      mbar_arm(ex.bar(b), (uint32_t)a.n_pad * 4u);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }

  load_rows_async(s.Gc, a.n_pad, a.G, a.ldg, r0, min(nr, a.cache), n, a.vec_ok != 0);
  const float v0 = rsqrtf((float)n);        // Lanczos start: all ones / sqrt(n)
  for (int i = e0; i < a.n_pad; i += nt) {
    const bool in = i < n;
    s.bb[i] = in ? a.b[i] : 0.f;
    s.x[i] = in ? a.x[i] : 0.f;
    s.y[i] = in ? v0 : 0.f;   // v_j
    s.z[i] = 0.f;             // v_{j-1}
  }
  cl.sync();   // every CTA's mbarriers are initialised and armed before any push

  // ---- Lipschitz constant: Lanczos (alpha = v^T G v, then beta = ||w||)
  float theta = 0.f, theta_prev = 0.f, beta_prev = 0.f;
  int m = 0;
  for (int j = 0; j < LZ_MAX; ++j) {
    float* Gv = cluster_gemv(a, s, s.y, r0, nr, ex, &s_bad);   // G v_j
    float va[1] = {0.f};
    for (int i = e0; i < n; i += nt) va[0] = fmaf(s.y[i], Gv[i], va[0]);
    block_sum_f<1>(va, s_red, parity);
    if (s_bad) {
      ok = false;
      break;
    }
    const float alpha = va[0];
    float vb[1] = {0.f};
    for (int i = e0; i < n; i += nt) {
      const float w = Gv[i] - alpha * s.y[i] - beta_prev * s.z[i];
      Gv[i] = w;
      vb[0] = fmaf(w, w, vb[0]);
    }
    block_sum_f<1>(vb, s_red, parity);
    const float beta = sqrtf(fmaxf(vb[0], 0.f));
    if (tid == 0) {
      s_al[j] = alpha;
      s_be[j] = beta;
    }
    m = j + 1;
    __syncthreads();
    const bool last = (m == n) || (m == LZ_MAX) || !(beta > 1e-7f * fabsf(alpha));
    if (last || (m % 4) == 0) {
      theta = tridiag_top(s_al, s_be, m, &s_theta);
      if (last || fabsf(theta - theta_prev) <= LZ_TOL * fabsf(theta)) break;
      theta_prev = theta;
    }
    const float inv = 1.f / beta;
    for (int i = e0; i < n; i += nt) {
      const float vn = Gv[i] * inv;
      s.z[i] = s.y[i];
      s.y[i] = vn;
    }
    beta_prev = beta;
    __syncthreads();
  }
  const float L = 1.01f * (theta > 0.f ? theta : 1.f);
  const float invL = 1.f / L;
  const float thr = __fmul_rn(a.lam, invL);

  // ---- initial G x
  if (ok) {
    const float* Gxr = cluster_gemv(a, s, s.x, r0, nr, ex, &s_bad);
    __syncthreads();
    ok = !s_bad;
    for (int i = e0; i < n; i += nt) {
      const float gx = Gxr[i];
      s.Gx[i] = gx;
      s.y[i] = s.x[i];
      s.Gy[i] = gx;
    }
  }

  // ---- monotone FISTA
  float t = 1.f;
  int it = 0;
  for (it = 1; it <= a.max_iter && ok; ++it) {
    for (int i = e0; i < n; i += nt) {
      const float u = s.y[i] - (s.Gy[i] - s.bb[i]) * invL;
      s.z[i] = (a.positive ? fmaxf(u - thr, 0.f) : copysignf(fmaxf(fabsf(u) - thr, 0.f), u));
    }
    __syncthreads();
    const float* Gz = cluster_gemv(a, s, s.z, r0, nr, ex, &s_bad);
    // F(z) - F(x) = sum_i (z_i - x_i) ((Gz_i + Gx_i) / 2 - b_i) + lambda (|z_i| - |x_i|)
    // (G symmetric): every term vanishes as z -> x, so an FP32 sum resolves the
    // sign of the difference where F itself (~1e7) would need ~50 bits
    float v[3] = {0.f, 0.f, 0.f};
    for (int i = e0; i < n; i += nt) {
      const float zr = s.z[i], xr = s.x[i];
      const float dF = fmaf(zr - xr, 0.5f * (Gz[i] + s.Gx[i]) - s.bb[i], a.lam * (fabsf(zr) - fabsf(xr)));
      v[0] += dF;
      const float d = zr - s.y[i];
      v[1] = fmaf(d, d, v[1]);
      v[2] = fmaf(zr, zr, v[2]);
    }
    const float t1 = 0.5f * (1.f + sqrtf(1.f + 4.f * t * t));
    const float c1 = t / t1, c2 = (t - 1.f) / t1;
    block_sum_f<3>(v, s_red, parity);
    if (s_bad) {
      ok = false;
      break;
    }
    const float step = sqrtf(v[1]);
    const float nz = sqrtf(v[2]);
    const bool accept = v[0] <= 0.f;
    for (int i = e0; i < n; i += nt) {
      const float xo = s.x[i], Gxo = s.Gx[i];
      const float xn = accept ? s.z[i] : xo;
      const float Gxn = accept ? Gz[i] : Gxo;
      s.y[i] = xn + c1 * (s.z[i] - xn) + c2 * (xn - xo);
      s.Gy[i] = Gxn + c1 * (Gz[i] - Gxn) + c2 * (Gxn - Gxo);
      s.x[i] = xn;
      s.Gx[i] = Gxn;
    }
    t = t1;
    if (step <= a.eps * nz) break;
  }
  if (it > a.max_iter) it = a.max_iter;
  // objective of the returned x, in double-float (reported only)
  Df Fx = {0.f, 0.f};
  if (ok) {
    Df v[NPART] = {};
    for (int i = e0; i < n; i += nt) {
      v[0] = df_add(v[0], df_prod(s.x[i], s.Gx[i]));
      v[1] = df_add(v[1], df_prod(s.bb[i], s.x[i]));
      v[2] = df_add(v[2], Df{fabsf(s.x[i]), 0.f});
    }
    block_sums(v, s_part, scratch);
    Fx = df_add(df_add(df_scale(s_part[0], 0.5f), df_neg(s_part[1])), df_scale(s_part[2], a.lam));
  }
  __syncthreads();
  if (ok) {
    for (int r = tid; r < nr; r += blockDim.x) a.x[r0 + r] = s.x[r0 + r];
    if (rank == 0 && tid == 0) {
      if (a.out_iters) *a.out_iters = it;
      if (a.out_L) *a.out_L = (double)L;
      if (a.out_F) *a.out_F = (double)Fx.hi + (double)Fx.lo;
      if (a.out_lanczos) *a.out_lanczos = m;
    }
  } else {
    // a wait expired: report it, and give pushes still addressed to this CTA
    // (bounded) time to land before it leaves
    if (tid == 0) {
      if (a.err) atomicExch(a.err, 1);
      mbar_wait_cluster(ex.bar(ex.buf), (ex.phase >> ex.buf) & 1u);
    }
    __syncthreads();
  }
  cl.sync();   // no CTA leaves while others may still address its shared memory
}

// ---------------------------------------------------------------------------
// Whole-GPU variant for supports whose G a cluster cannot keep on the chip: the
// iteration of k_apgd_full (every CTA keeps the vectors whole and owns a block of
// rows of G, the same sums in the same order, hence the same results) over up to
// one CTA per SM, so that G stays in shared memory. Vectors live in registers
// (thread i holds entries i + 256 k). A product's entries go to all CTAs through
// global memory as 64-bit words, the value and the product's number: a reader
// polls the words themselves, so that an exchange costs one write and one read of
// L2 and needs no barrier, fence or flag.
//
// A warp takes four rows and writes their words with one instruction, a whole
// 32-byte sector: sectors written in parts, while every CTA polls them, made an
// iteration 5 to 8 us instead of 2.3 to 4 (900 to 2500 atoms; 8 to 24 rows a CTA
// against 32; pauses between the polls gained nothing). All of a thread's words
// are asked for together.
//
// Two mailboxes alternate. A CTA writes product i + 2 only after reading all of
// product i + 1, each entry of which was written after its CTA had read all of
// product i, so no entry is overwritten while it is awaited. The launch is
// cooperative (all CTAs resident); every wait has a limit.
//
// What bounds it: the latency of the exchange. Measured against k_apgd_full on 16
// SMs, us an iteration: 900 atoms 3.8 and 2.8, 1300 5.7 and 2.7, 1700 8.1 and 3.0,
// 2500 16.0 and 3.8.
constexpr int GRID_THREADS = 256;
constexpr int GRID_EMAX = 12;                       // entries per thread: supports of up to 3072
constexpr int GRID_ROWS = 32;                       // rows per CTA at most: four a warp (a multiple of 4)

__device__ __forceinline__ void mail_put(unsigned long long* p, unsigned tag, float v) {
  const unsigned long long w = ((unsigned long long)tag << 32) | __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}
__device__ __forceinline__ unsigned long long mail_get(const unsigned long long* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return w;
}

template <int E>   // entries per thread
__global__ void __launch_bounds__(GRID_THREADS, 1) k_apgd_grid(const __grid_constant__ ApgdArgs a,
                                                              unsigned long long* __restrict__ mail) {
  extern __shared__ __align__(16) float apgdg_sm[];   // the input vector (n_pad), rows of G
  __shared__ Df scratch[(GRID_THREADS / 32) * NPART];
  __shared__ Df s_part[NPART];
  __shared__ __align__(16) float s_red[2][3][8];
  __shared__ float s_al[LZ_MAX], s_be[LZ_MAX], s_theta;
  __shared__ int s_bad;
  float* vec_s = apgdg_sm;
  float* Gc = apgdg_sm + a.n_pad;
  const int n = a.n, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r0 = (int)blockIdx.x * a.rows_per;
  const int nr = max(0, min(n, r0 + a.rows_per) - r0);
  const bool vecld = !a.scalar;
  unsigned tag = 0;
  int parity = 0;

  load_rows_async(Gc, a.n_pad, a.G, a.ldg, r0, nr, n, a.vec_ok != 0);
  for (int i = n + tid; i < a.n_pad; i += GRID_THREADS) vec_s[i] = 0.f;
  if (tid == 0) s_bad = 0;
  const float v0 = rsqrtf((float)n);        // Lanczos start: all ones / sqrt(n)
  float x[E], Gx[E], y[E], Gy[E], bb[E], z[E], Gz[E];
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const int i = tid + GRID_THREADS * k;
    bb[k] = i < n ? a.b[i] : 0.f;
    x[k] = i < n ? a.x[i] : 0.f;
    y[k] = i < n ? v0 : 0.f;   // v_j
    z[k] = 0.f;                // v_{j-1}
  }

  // out = G in, every CTA all of it. A wait that expires leaves s_bad set for the
  // caller to read behind its next barrier. The caller's barrier since the last
  // product has ended every read of vec_s.
  auto product = [&](const float (&in)[E], float (&out)[E]) {
#pragma unroll
    for (int k = 0; k < E; ++k) {
      const int i = tid + GRID_THREADS * k;
      if (i < n) vec_s[i] = in[k];
    }
    __syncthreads();
    ++tag;
    unsigned long long* box = mail + (size_t)(tag & 1u) * a.n_pad;
    for (int rb = 4 * warp; rb < nr; rb += 4 * (GRID_THREADS / 32)) {
      const float* rows[4];
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int q = 0; q < 4; ++q) rows[q] = Gc + (size_t)min(rb + q, nr - 1) * a.n_pad;
      rows_dot<4>(rows, vec_s, n, !a.scalar, acc);
      for (int off = 16; off; off >>= 1)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], off);
      if (lane < min(4, nr - rb))                     // 32 bytes: a whole sector
        mail_put(box + r0 + rb + lane, tag, lane & 2 ? (lane & 1 ? acc[3] : acc[2]) : (lane & 1 ? acc[1] : acc[0]));
    }
    // all entries asked for at once, those that had not come once more
    unsigned long long w[E];
    const long long t0 = clock64();
    bool good = true, all;
#pragma unroll
    for (int k = 0; k < E; ++k) w[k] = tid + GRID_THREADS * k < n ? 0ull : (unsigned long long)tag << 32;
    do {
      all = true;
#pragma unroll
      for (int k = 0; k < E; ++k)
        if ((unsigned)(w[k] >> 32) != tag) w[k] = mail_get(box + tid + GRID_THREADS * k);
#pragma unroll
      for (int k = 0; k < E; ++k) all = all && (unsigned)(w[k] >> 32) == tag;
      good = all || clock64() - t0 <= APGD_WAIT_CYCLES;
    } while (!all && good);
#pragma unroll
    for (int k = 0; k < E; ++k) out[k] = __uint_as_float((unsigned)w[k]);
    if (!good) s_bad = 1;
  };

  // ---- Lipschitz constant: Lanczos (alpha = v^T G v, then beta = ||w||)
  float theta = 0.f, theta_prev = 0.f, beta_prev = 0.f;
  int m = 0;
  bool ok = true;
  __syncthreads();
  for (int j = 0; j < LZ_MAX; ++j) {
    product(y, Gz);
    float va[1] = {0.f};
#pragma unroll
    for (int k = 0; k < E; ++k)
      if (tid + GRID_THREADS * k < n) va[0] = fmaf(y[k], Gz[k], va[0]);
    block_sum_f<1>(va, s_red, parity);
    if (s_bad) {
      ok = false;
      break;
    }
    const float alpha = va[0];
    float vb[1] = {0.f};
#pragma unroll
    for (int k = 0; k < E; ++k)
      if (tid + GRID_THREADS * k < n) {
        const float w = Gz[k] - alpha * y[k] - beta_prev * z[k];
        Gz[k] = w;
        vb[0] = fmaf(w, w, vb[0]);
      }
    block_sum_f<1>(vb, s_red, parity);
    const float beta = sqrtf(fmaxf(vb[0], 0.f));
    if (tid == 0) {
      s_al[j] = alpha;
      s_be[j] = beta;
    }
    m = j + 1;
    __syncthreads();
    const bool last = (m == n) || (m == LZ_MAX) || !(beta > 1e-7f * fabsf(alpha));
    if (last || (m % 4) == 0) {
      theta = tridiag_top(s_al, s_be, m, &s_theta);
      if (last || fabsf(theta - theta_prev) <= LZ_TOL * fabsf(theta)) break;
      theta_prev = theta;
    }
    const float inv = 1.f / beta;
#pragma unroll
    for (int k = 0; k < E; ++k) {
      z[k] = y[k];
      y[k] = Gz[k] * inv;
    }
    beta_prev = beta;
  }
  const float L = 1.01f * (theta > 0.f ? theta : 1.f);
  const float invL = 1.f / L;
  const float thr = __fmul_rn(a.lam, invL);

  // ---- initial G x
  if (ok) {
    product(x, Gx);
    __syncthreads();
    ok = !s_bad;
#pragma unroll
    for (int k = 0; k < E; ++k) {
      y[k] = x[k];
      Gy[k] = Gx[k];
    }
  }

  // ---- monotone FISTA
  float t = 1.f;
  int it = 0;
  for (it = 1; it <= a.max_iter && ok; ++it) {
#pragma unroll
    for (int k = 0; k < E; ++k) {
      const float u = y[k] - (Gy[k] - bb[k]) * invL;
      z[k] = (a.positive ? fmaxf(u - thr, 0.f) : copysignf(fmaxf(fabsf(u) - thr, 0.f), u));
    }
    product(z, Gz);
    // F(z) - F(x) from the difference itself (see k_apgd_full)
    float v[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < E; ++k)
      if (tid + GRID_THREADS * k < n) {
        const float dF =
            fmaf(z[k] - x[k], 0.5f * (Gz[k] + Gx[k]) - bb[k], a.lam * (fabsf(z[k]) - fabsf(x[k])));
        v[0] += dF;
        const float d = z[k] - y[k];
        v[1] = fmaf(d, d, v[1]);
        v[2] = fmaf(z[k], z[k], v[2]);
      }
    const float t1 = 0.5f * (1.f + sqrtf(1.f + 4.f * t * t));
    const float c1 = t / t1, c2 = (t - 1.f) / t1;
    block_sum_f<3>(v, s_red, parity);
    if (s_bad) {
      ok = false;
      break;
    }
    const float step = sqrtf(v[1]);
    const float nz = sqrtf(v[2]);
    const bool accept = v[0] <= 0.f;
#pragma unroll
    for (int k = 0; k < E; ++k) {
      const float xo = x[k], Gxo = Gx[k];
      const float xn = accept ? z[k] : xo;
      const float Gxn = accept ? Gz[k] : Gxo;
      y[k] = xn + c1 * (z[k] - xn) + c2 * (xn - xo);
      Gy[k] = Gxn + c1 * (Gz[k] - Gxn) + c2 * (Gxn - Gxo);
      x[k] = xn;
      Gx[k] = Gxn;
    }
    t = t1;
    if (step <= a.eps * nz) break;
  }
  if (it > a.max_iter) it = a.max_iter;
  if (!ok) {
    if (tid == 0 && a.err) atomicExch(a.err, 1);
    return;
  }
#pragma unroll
  for (int k = 0; k < E; ++k) {
    const int i = tid + GRID_THREADS * k;
    if (i >= r0 && i < r0 + nr) a.x[i] = x[k];
  }
  if (blockIdx.x != 0) return;
  // objective of the returned x, in double-float (reported only)
  Df p[NPART] = {};
#pragma unroll
  for (int k = 0; k < E; ++k) {
    p[0] = df_add(p[0], df_prod(x[k], Gx[k]));
    p[1] = df_add(p[1], df_prod(bb[k], x[k]));
    p[2] = df_add(p[2], Df{fabsf(x[k]), 0.f});
  }
  block_sums(p, s_part, scratch);
  if (tid == 0) {
    const Df Fx = df_add(df_add(df_scale(s_part[0], 0.5f), df_neg(s_part[1])), df_scale(s_part[2], a.lam));
    if (a.out_iters) *a.out_iters = it;
    if (a.out_L) *a.out_L = (double)L;
    if (a.out_F) *a.out_F = (double)Fx.hi + (double)Fx.lo;
    if (a.out_lanczos) *a.out_lanczos = m;
  }
}

// ---------------------------------------------------------------------------
// One-CTA variant for supports of up to CTA_NMAX atoms: the same Lanczos step
// size, monotone FISTA, stop rule and reported objective, with two threads per
// row of G and of every vector. Thread h of a row's two holds the row's columns
// 4 c + 2 h and 4 c + 2 h + 1 in registers (the last NS of its columns in shared
// memory where the block's threads leave too few registers) and sums each of the
// two series in the order of c; a product reads only the broadcast vector. An
// iteration is a serial chain of two block barriers (input vector complete;
// partial sums complete), the product and the sums, so everything else is kept
// off it: one further warp evaluates the momentum's coefficients during the
// product and the stop test during the next proximal step, which a stop discards.
// Measured against a thread per row with G in shared memory (and one warp for
// the whole problem up to 64 atoms), us an iteration before and after: 40 atoms
// 0.66 and 0.50, 120 1.09 and 0.60, 160 1.31 and 1.03, 224 1.83 and 1.28.
//
// Order of the sums: a warp holds 16 rows, every second of 32 consecutive ones
// (SMALL: every fourth of all 64, rows r and r + 32 first), so that the sums over
// a warp and then over the warps of a group add as a butterfly over 32 rows (64)
// does; groups of 32 follow in turn.
constexpr int WARP_NMAX = 64;    // one tree over all rows
constexpr int CTA_NMAX = 224;

__device__ __forceinline__ float pair_butterfly(float t, bool from_first) {
  if (from_first) t += __shfl_xor_sync(0xffffffffu, t, 16);
  t += __shfl_xor_sync(0xffffffffu, t, 8);
  t += __shfl_xor_sync(0xffffffffu, t, 4);
  t += __shfl_xor_sync(0xffffffffu, t, 2);
  return t;
}

// sum over rows of a b (SMALL: a fused multiply-add per pair of rows r, r + 32)
template <bool SMALL>
__device__ __forceinline__ float pair_product_sum(float a, float b) {
  const float p = __fmul_rn(a, b);
  if (!SMALL) return pair_butterfly(p, true);
  return pair_butterfly(fmaf(a, b, __shfl_xor_sync(0xffffffffu, p, 16)), false);
}

// block-wide total of the warps' partial sums red[0..)
template <int GROUPS>
__device__ __forceinline__ float pair_total(const float* red) {
  const float4* p = reinterpret_cast<const float4*>(red);
  if (GROUPS == 0) {                                // SMALL: four warps, one tree
    const float4 f = p[0];
    return (f.x + f.z) + (f.y + f.w);
  }
  float t = 0.f;
#pragma unroll
  for (int g = 0; g < GROUPS; g += 2) {             // zeros past the last group
    const float4 f = p[g >> 1];
    t += f.x + f.y;
    t += f.z + f.w;
  }
  return t;
}

template <int NC, int NS>   // columns per thread (n <= 2 NC), the last NS of them in shared memory
__global__ void __launch_bounds__(4 * NC + 32, 1) k_apgd_cta(const __grid_constant__ ApgdBatch batch) {
  constexpr bool SMALL = 2 * NC <= WARP_NMAX;
  constexpr int GROUPS = SMALL ? 0 : (2 * NC + 31) / 32;
  constexpr int NR = NC - NS, LDV = NC + 4;         // LDV: the halves of vs in different banks
  extern __shared__ __align__(16) float4 apgdc_sm[];   // NS / 4 x threads
  __shared__ __align__(16) float vs[2 * LDV];       // the broadcast input: entry i at [i % 4 / 2][i / 4 * 2 + i % 2]
  __shared__ __align__(16) float s_red[2][3][16];   // [buffer][value][warp]
  __shared__ float2 s_mom;                          // momentum coefficients of the iteration
  __shared__ int s_stop;
  __shared__ Df s_dred[16 * 3];
  __shared__ float s_al[LZ_MAX], s_be[LZ_MAX], s_theta;
  const ApgdArgs& a = batch.job[blockIdx.x];
  const int n = a.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int threads = blockDim.x - 32;              // the last warp holds no rows
  const int groups = threads >> 6, h = lane & 1;
  const bool rows_warp = tid < threads;
  const int row = SMALL ? warp + 4 * (lane >> 1) : 32 * (warp >> 1) + (warp & 1) + 2 * (lane >> 1);
  const int slot = rows_warp ? tid : 0;             // of apgdc_sm: the last warp has none of its own
  const bool own = rows_warp && row < n, put = own && h == 0;
  float* vrow = vs + ((row & 2) ? LDV : 0) + (row >> 2) * 2 + (row & 1);
  float g[NR];
  {
    const float* src = a.G + (size_t)(own ? row : 0) * a.ldg;
    auto at = [&](int e) {                          // this thread's e-th column
      const int c = 4 * (e >> 1) + 2 * h + (e & 1);
      return own && c < n ? src[c] : 0.f;
    };
#pragma unroll
    for (int e = 0; e < NR; ++e) g[e] = at(e);
    if (NS && rows_warp)
#pragma unroll
      for (int e = 0; e < NS; e += 4)
        apgdc_sm[e / 4 * threads + tid] = make_float4(at(NR + e), at(NR + e + 1), at(NR + e + 2), at(NR + e + 3));
  }
  auto product = [&]() {
    const float4* v4 = reinterpret_cast<const float4*>(vs + h * LDV);
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int e = 0; e < NR; e += 4) {               // zeros past n: a test per step would keep
      const float4 z = v4[e / 4];                   // the loads from overlapping
      a0 = fmaf(g[e], z.x, a0);
      a1 = fmaf(g[e + 1], z.y, a1);
      a0 = fmaf(g[e + 2], z.z, a0);
      a1 = fmaf(g[e + 3], z.w, a1);
    }
#pragma unroll
    for (int e = 0; e < NS; e += 4) {
      const float4 z = v4[(NR + e) / 4], f = apgdc_sm[e / 4 * threads + slot];
      a0 = fmaf(f.x, z.x, a0);
      a1 = fmaf(f.y, z.y, a1);
      a0 = fmaf(f.z, z.z, a0);
      a1 = fmaf(f.w, z.w, a1);
    }
    float t = a0 + a1;
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    return own ? t : 0.f;
  };
  const float bb = own ? a.b[row] : 0.f;
  float x = own ? a.x[row] : 0.f;
  int parity = 0;
  // one sum over the rows of p q, the same in every thread
  auto block_product_sum = [&](float p, float q) {
    const float t = pair_product_sum<SMALL>(p, q);
    if (rows_warp && lane == 0) s_red[parity][0][warp] = t;
    __syncthreads();
    const float r = pair_total<GROUPS>(s_red[parity][0]);
    parity ^= 1;
    return r;
  };

  // ---- Lipschitz constant: Lanczos from the all-ones vector
  float v = own ? rsqrtf((float)n) : 0.f, vprev = 0.f;
  for (int i = tid; i < 2 * LDV; i += blockDim.x) vs[i] = 0.f;
  for (int i = tid; i < 2 * 3 * 16; i += blockDim.x) (&s_red[0][0][0])[i] = 0.f;
  __syncthreads();
  if (put) *vrow = v;
  __syncthreads();
  float theta = 0.f, theta_prev = 0.f, beta_prev = 0.f;
  int m = 0;
  for (int j = 0; j < LZ_MAX; ++j) {
    const float gv = product();
    const float alpha = block_product_sum(v, gv);
    const float w = own ? gv - alpha * v - beta_prev * vprev : 0.f;
    const float beta = sqrtf(fmaxf(block_product_sum(w, w), 0.f));
    if (tid == 0) {
      s_al[j] = alpha;
      s_be[j] = beta;
    }
    m = j + 1;
    const bool last = (m == n) || (m == LZ_MAX) || !(beta > 1e-7f * fabsf(alpha));
    if (last || (m % 4) == 0) {
      __syncthreads();                              // s_al, s_be written
      theta = tridiag_top(s_al, s_be, m, &s_theta);
      if (last || fabsf(theta - theta_prev) <= LZ_TOL * fabsf(theta)) break;
      theta_prev = theta;
    }
    vprev = v;
    v = SMALL ? w * (1.f / beta) : w / beta;
    if (put) *vrow = v;                             // every read of vs ended before the sums
    beta_prev = beta;
    __syncthreads();
  }
  const float L = 1.01f * (theta > 0.f ? theta : 1.f);
  const float invL = 1.f / L;
  const float thr = __fmul_rn(a.lam, invL);
  // |u| - lambda / L, in SMALL with one rounding
  auto shrink = [&](float v) { return fmaxf(SMALL ? fmaf(-a.lam, invL, v) : v - thr, 0.f); };

  // ---- initial G x
  __syncthreads();                                  // every read of vs ended
  if (put) *vrow = x;
  if (tid == 0) s_stop = 0;
  __syncthreads();
  float Gx = product();
  float y = x, Gy = Gx;
  __syncthreads();                                  // every read of vs ended

  // ---- monotone FISTA
  float t = 1.f;                                    // the last warp's: momentum
  int it = 0;
  for (it = 1; it <= a.max_iter; ++it) {
    const float u = y - (Gy - bb) * invL;
    float z = a.positive ? shrink(u) : copysignf(shrink(fabsf(u)), u);
    if (!own) z = 0.f;
    if (put) *vrow = z;                             // the last product's reads ended before its sums
    __syncthreads();
    if (s_stop) break;                              // the iteration before was the last one
    float Gz = 0.f;
    if (rows_warp) {
      Gz = product();
      // F(z) - F(x) from the difference itself (see k_apgd_full); the row's two
      // threads take a sum each, and share the third
      const float d = z - y;
      const float dF = own ? fmaf(z - x, 0.5f * (Gz + Gx) - bb, a.lam * (fabsf(z) - fabsf(x))) : 0.f;
      const float dd = __fmul_rn(d, d);
      float r0;
      if (SMALL) {
        const float o = __shfl_xor_sync(0xffffffffu, h ? dd : dF, 16);
        r0 = pair_butterfly(h ? fmaf(d, d, o) : dF + o, false);
      } else {
        r0 = pair_butterfly(h ? dd : dF, true);
      }
      const float r2 = pair_product_sum<SMALL>(z, z);
      if (lane < 2) s_red[parity][h][warp] = r0;
      if (lane == 0) s_red[parity][2][warp] = r2;
    } else if (lane == 0) {
      const float t1 = 0.5f * (1.f + sqrtf(1.f + 4.f * t * t));
      s_mom = make_float2(t / t1, (t - 1.f) / t1);
      t = t1;
    }
    __syncthreads();
    if (rows_warp) {
      const bool accept = pair_total<GROUPS>(s_red[parity][0]) <= 0.f;
      const float c1 = s_mom.x, c2 = s_mom.y;
      const float xn = accept ? z : x, Gxn = accept ? Gz : Gx;
      y = xn + c1 * (z - xn) + c2 * (xn - x);
      Gy = Gxn + c1 * (Gz - Gxn) + c2 * (Gxn - Gx);
      x = xn;
      Gx = Gxn;
    } else if (lane == 0) {
      const float step = sqrtf(pair_total<GROUPS>(s_red[parity][1]));
      const float nz = sqrtf(pair_total<GROUPS>(s_red[parity][2]));
      s_stop = step <= a.eps * nz;
    }
    parity ^= 1;
  }
  it = min(it - 1, a.max_iter);
  // objective of the returned x, in double-float (reported only)
  {
    Df p[3] = {df_prod(x, Gx), df_prod(bb, x), Df{fabsf(x), 0.f}};
    for (int off = 16; off > 1; off >>= 1)
#pragma unroll
      for (int i = 0; i < 3; ++i) p[i] = df_add(p[i], df_shfl_xor(p[i], off));
    if (rows_warp && lane == 0)
#pragma unroll
      for (int i = 0; i < 3; ++i) s_dred[warp * 3 + i] = p[i];
    __syncthreads();
    if (tid == 0) {
      Df tot[3] = {};
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (SMALL)
          tot[i] = df_add(df_add(s_dred[i], s_dred[6 + i]), df_add(s_dred[3 + i], s_dred[9 + i]));
        else
          for (int w = 0; w < 2 * groups; w += 2)
            tot[i] = df_add(tot[i], df_add(s_dred[w * 3 + i], s_dred[w * 3 + 3 + i]));
      }
      const Df Fx = df_add(df_add(df_scale(tot[0], 0.5f), df_neg(tot[1])), df_scale(tot[2], a.lam));
      if (a.out_iters) *a.out_iters = it;
      if (a.out_L) *a.out_L = (double)L;
      if (a.out_F) *a.out_F = (double)Fx.hi + (double)Fx.lo;
      if (a.out_lanczos) *a.out_lanczos = m;
    }
  }
  if (put) a.x[row] = x;
}

// Columns per thread of each instantiation. Registers: 65536 over the block's
// threads; the largest keeps its last columns in shared memory.
constexpr int CTA_NC[4] = {32, 64, 96, 112};
constexpr int CTA_NS = 16;

}  // namespace

namespace {

// Launch shape of one restricted problem: which kernel, cluster size, rows per
// CTA, whether the CTAs cache their rows of G, dynamic shared memory.
struct ApgdShape {
  int cta = -1;        // one-CTA kernel (n <= CTA_NMAX): its instantiation (CTA_NC)
  bool full;
  int CS;
  int rows_per;
  int cache;
  int n_pad;
  size_t smem;
  int threads = APGD_THREADS;
  bool by_alignment = false;   // unaligned rows of G by single columns
  int grid = 0;        // whole-GPU kernel: its CTAs
};

// dynamic shared memory ceilings: 227 KB per CTA minus the kernels' static arrays
constexpr size_t kLimitRows = 200 * 1024;
constexpr size_t kLimitFull = 231200;
constexpr size_t kLimitGrid = 224 * 1024;

int apgd_setup(int* cs_max_out) {
  static int cs_max = 0;
  static bool attrs_set = false;
  if (cs_max == 0) {
    cudaError_t e1 = cudaFuncSetAttribute(k_apgd, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaError_t e2 = cudaFuncSetAttribute(k_apgd_full<APGD_THREADS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cudaError_t e3 =
        cudaFuncSetAttribute(k_apgd_full<2 * APGD_THREADS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    cs_max = (e1 == cudaSuccess && e2 == cudaSuccess && e3 == cudaSuccess) ? 16 : 8;
    cudaGetLastError();
  }
  if (!attrs_set) {
    PC_CUDA(cudaFuncSetAttribute(k_apgd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLimitRows));
    PC_CUDA(cudaFuncSetAttribute(k_apgd_full<APGD_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kLimitFull));
    PC_CUDA(cudaFuncSetAttribute(k_apgd_full<2 * APGD_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kLimitFull));
    PC_CUDA(cudaFuncSetAttribute(k_apgd_grid<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLimitGrid));
    PC_CUDA(cudaFuncSetAttribute(k_apgd_grid<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLimitGrid));
    PC_CUDA(cudaFuncSetAttribute(k_apgd_grid<GRID_EMAX>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kLimitGrid));
    attrs_set = true;
  }
  *cs_max_out = cs_max;
  return PC_OK;
}

int apgd_shape(int S, int cs_max, ApgdShape* out) {
  const int n_pad = (S + 3) & ~3;
  // full-vector kernel: 2 receive buffers and 6 full vectors, and as many rows of
  // G as fit beside them; a CTA's rows are a multiple of 4 (16-byte stores)
  auto rows_full = [&](int cs) { return cluster_rows(S, cs); };
  const size_t vec_full = sizeof(float) * 8 * (size_t)n_pad, row_full = sizeof(float) * (size_t)n_pad;
  // row-slice kernel (larger supports): one full vector + 8 row slices
  auto bytes_rows = [&](int cs, bool cached) {
    const size_t rp = (size_t)ceil_div(S, cs);
    return sizeof(float) * ((size_t)n_pad + 8 * rp) + 16 + 16 * sizeof(Df) +
           (cached ? sizeof(float) * rp * n_pad : 0);
  };
  // cluster size: the smallest power of two whose CTAs each hold at most 32 KB of
  // G (a matrix-vector product then streams it in ~250 cycles), else cs_max
  ApgdShape sh;
  if (S <= CTA_NMAX) {
    sh.cta = 0;
    while (S > 2 * CTA_NC[sh.cta]) ++sh.cta;
    sh.full = true;
    sh.CS = 1;
    sh.cache = 1;
    sh.smem = 0;
    sh.rows_per = S;
    sh.n_pad = n_pad;
    *out = sh;
    return PC_OK;
  }
  sh.full = true;
  sh.CS = 1;
  const size_t share_target = 32 * 1024;
  while (sh.CS < cs_max && rows_full(sh.CS) * row_full > share_target) sh.CS *= 2;
  // rows of G in shared memory: all, else as many as fit if that is half of them,
  // else 170 KB, which leaves the rows read from L2 a first-level cache to arrive in
  // (2500 atoms, 225 KB: 19.6 us an iteration, 170 KB 16.0; 900 atoms 3.76 and 4.09).
  // With rows to read 16 warps multiply, not 8 (1300 atoms 6.6 and 5.7 us).
  auto fit = [&](size_t lim) { return lim > vec_full ? (int)((lim - vec_full) / row_full) & ~3 : 0; };
  const int rp = rows_full(sh.CS);
  sh.cache = std::min(rp, fit(kLimitFull));
  if (sh.cache < rp) {
    sh.threads = 2 * APGD_THREADS;
    if (2 * sh.cache < rp) sh.cache = fit(170 * 1024);
    // a lane's columns, hence the order of its sum, go by the alignment of the rows
    // unless 226 KB hold all of them beside the vectors and two slices
    sh.by_alignment = 2 * sizeof(float) * rp + vec_full + rp * row_full > 226 * 1024;
  }
  sh.smem = vec_full + sh.cache * row_full;
  if (2 * sizeof(float) * rp + vec_full > 226 * 1024) {
    sh.full = false;
    sh.threads = APGD_THREADS;
    sh.by_alignment = false;
    sh.CS = 1;
    while (sh.CS < cs_max && bytes_rows(sh.CS, true) > kLimitRows) sh.CS *= 2;
    if (bytes_rows(sh.CS, false) > kLimitRows)
      return fail(PC_ERR_CAPACITY, "apgd: support of %d atoms exceeds the cluster solver", S);
    sh.cache = bytes_rows(sh.CS, true) <= kLimitRows ? 1 : 0;
    sh.smem = bytes_rows(sh.CS, sh.cache != 0);
  }
  sh.rows_per = sh.full ? rows_full(sh.CS) : ceil_div(S, sh.CS);
  sh.n_pad = n_pad;
  *out = sh;
  return PC_OK;
}

ApgdArgs make_args(const ApgdJob& j, const ApgdShape& sh) {
  ApgdArgs a;
  a.G = j.G;
  a.ldg = j.ldg;
  a.b = j.b;
  a.n = j.n;
  a.lam = (float)j.lambda;
  a.eps = (float)j.eps;
  a.max_iter = j.max_iter;
  a.x = j.x;
  a.out_iters = j.iters;
  a.out_L = j.L;
  a.out_F = j.F;
  a.out_lanczos = j.lanczos;
  a.err = j.err;
  a.positive = j.positive ? 1 : 0;
  a.rows_per = sh.rows_per;
  a.n_pad = sh.n_pad;
  a.cache = sh.cache;
  a.vec_ok = ((j.ldg & 3) == 0 && (reinterpret_cast<uintptr_t>(j.G) & 15) == 0) ? 1 : 0;
  a.scalar = sh.by_alignment && !a.vec_ok;
  return a;
}

}  // namespace

// Whole-GPU shape of a support whose G a cluster would read from L2 (cl: its cluster
// shape): from about 870 atoms, where the cluster is the slower one (us an iteration,
// 700 atoms 2.5 on the cluster and 2.4, 900 3.8 and 2.8, 1300 5.7 and 2.7), to about
// 2750, where one CTA per SM no longer holds all rows.
static bool apgd_grid_shape(int S, const ApgdShape& cl, ApgdShape* sh) {
  if (!cl.full || cl.cta >= 0 || cl.cache >= cl.rows_per || S > GRID_THREADS * GRID_EMAX) return false;
  int dev = 0, n_sm = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  if (!coop || n_sm < 1) return false;
  *sh = cl;
  const size_t row = sizeof(float) * (size_t)sh->n_pad;
  sh->rows_per = std::min(GRID_ROWS, (int)(kLimitGrid / row - 1) & ~3);
  if (sh->rows_per < 4) return false;
  sh->grid = ceil_div(S, sh->rows_per);
  sh->cache = sh->rows_per;
  sh->smem = row * (1 + sh->rows_per);
  return sh->grid <= n_sm;
}

static int launch_apgd_grid(const ApgdJob& j, const ApgdShape& sh, unsigned long long* mail, cudaStream_t st) {
  PC_CUDA(cudaMemsetAsync(mail, 0, 2 * sizeof(*mail) * (size_t)sh.n_pad, st));   // product numbers start at 1
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sh.grid, 1, 1);
  cfg.blockDim = dim3(GRID_THREADS, 1, 1);
  cfg.dynamicSmemBytes = sh.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const ApgdArgs a = make_args(j, sh);
  ProfScope prof_scope_(PROF_APGD, st);
  prof_scope_.kernels = 1;
  PC_CUDA(j.n <= 4 * GRID_THREADS   ? cudaLaunchKernelEx(&cfg, k_apgd_grid<4>, a, mail)
          : j.n <= 8 * GRID_THREADS ? cudaLaunchKernelEx(&cfg, k_apgd_grid<8>, a, mail)
                                    : cudaLaunchKernelEx(&cfg, k_apgd_grid<GRID_EMAX>, a, mail));
  return PC_OK;
}

int run_apgd_jobs(const ApgdJob* jobs, int n_jobs, cudaStream_t st) {
  int cs_max = 0;
  PC_TRY(apgd_setup(&cs_max));
  // a support alone may take the whole GPU; several run side by side on their clusters
  if (n_jobs == 1 && jobs[0].n > 0) {
    ApgdShape cl, one;
    PC_TRY(apgd_shape(jobs[0].n, cs_max, &cl));
    void* mail = nullptr;
    if (apgd_grid_shape(jobs[0].n, cl, &one)) {
      if (dmalloc(&mail, 2 * sizeof(unsigned long long) * (size_t)one.n_pad, st) == PC_OK) {
        const int rc = launch_apgd_grid(jobs[0], one, static_cast<unsigned long long*>(mail), st);
        dfree(mail, st);
        return rc;
      }
      clear_error();                        // no room: the cluster needs none
    }
  }
  std::vector<ApgdShape> shapes(n_jobs);
  for (int i = 0; i < n_jobs; ++i)
    if (jobs[i].n > 0) PC_TRY(apgd_shape(jobs[i].n, cs_max, &shapes[i]));
  std::vector<char> done(n_jobs, 0);
  for (int i = 0; i < n_jobs; ++i)
    if (jobs[i].n <= 0) done[i] = 1;
  // one launch per (kernel, cluster size) group, at most APGD_BATCH_MAX jobs each
  for (int i = 0; i < n_jobs; ++i) {
    if (done[i]) continue;
    ApgdBatch batch{};
    size_t smem = 0;
    const bool full = shapes[i].full;
    const int cta = shapes[i].cta;
    int rows = 0;
    const int CS = shapes[i].CS;
    for (int j = i; j < n_jobs && batch.n_jobs < APGD_BATCH_MAX; ++j) {
      if (done[j] || shapes[j].full != full || shapes[j].CS != CS || shapes[j].cta != cta ||
          shapes[j].threads != shapes[i].threads)
        continue;
      batch.job[batch.n_jobs++] = make_args(jobs[j], shapes[j]);
      smem = std::max(smem, shapes[j].smem);
      rows = std::max(rows, jobs[j].n);
      done[j] = 1;
    }
    if (cta >= 0) {
      ProfScope prof_scope_(PROF_APGD, st);
      prof_scope_.kernels = 1;
      // two threads a row, whole groups of 32 rows (64 of the smallest), and the last warp
      const int rt = cta == 0 ? 2 * WARP_NMAX : 64 * ceil_div(rows, 32), threads = rt + 32;
      if (cta == 0)
        k_apgd_cta<CTA_NC[0], 0><<<batch.n_jobs, threads, 0, st>>>(batch);
      else if (cta == 1)
        k_apgd_cta<CTA_NC[1], 0><<<batch.n_jobs, threads, 0, st>>>(batch);
      else if (cta == 2)
        k_apgd_cta<CTA_NC[2], 0><<<batch.n_jobs, threads, 0, st>>>(batch);
      else
        k_apgd_cta<CTA_NC[3], CTA_NS><<<batch.n_jobs, threads, sizeof(float) * CTA_NS * rt, st>>>(batch);
      PC_LAUNCH_CHECK();
      continue;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS * batch.n_jobs, 1, 1);
    cfg.blockDim = dim3(shapes[i].threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    {
      ProfScope prof_scope_(PROF_APGD, st);
      prof_scope_.kernels = 1;
      e = !full                                ? cudaLaunchKernelEx(&cfg, k_apgd, batch)
          : shapes[i].threads == APGD_THREADS ? cudaLaunchKernelEx(&cfg, k_apgd_full<APGD_THREADS>, batch)
                                              : cudaLaunchKernelEx(&cfg, k_apgd_full<2 * APGD_THREADS>, batch);
    }
    PC_CUDA(e);
  }
  return PC_OK;
}

int run_apgd(const float* G, int ldg, const float* b, int S, double lambda, double eps,
             int max_iter, float* x, int* iters, double* L, double* Fx, cudaStream_t st,
             int* lanczos, int* err, bool positive) {
  if (S <= 0) return PC_OK;
  ApgdJob j{G, ldg, b, S, lambda, eps, max_iter, x, iters, L, Fx, lanczos, err, positive};
  return run_apgd_jobs(&j, 1, st);
}

}  // namespace pc
