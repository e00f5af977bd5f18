// Transforms at the resolution of the visibilities.
//
// An image is usually sampled finer than its visibilities resolve: a source's
// response turns |u| dl times per pixel, 0.08 to 0.28 in the configurations, where
// the image could hold 0.5. The w-plane transforms then run on a smaller image of
// the same field (side Nt = G / 2, pixels d times wider, so the grid's side G is
// 2 to 4 times smaller and its cells stay as wide as they were), and the sum of
// the planes, corrected and real, is interpolated to the N x N pixels:
//
//   img[i][j] = sum_{k, l < K} g(x_i - k) g(x_j - l) small[k][l],  x_i = (i - N/2) / d + Nt/2,
//   g(x) = sinc(x) I0(beta sqrt(1 - (2x/K)^2)) / I0(beta),  beta = pi K (1/2 - nu),
//
// the Kaiser-windowed sinc, for a band |frequency| <= nu cycles per small pixel
// (nu from max |u|, |v| and the slope of the w-term, which climbs over the taps). With
// beta >= 15.1, the rule's bound, it is within 1.5e-7 (rms 5e-8) of e^{2 pi i f x} over
// the band and within 2.1e-7 of a wave whose frequency climbs: a tenth of the
// operators' own error on the border. The forward operator runs the
// transpose.
//
// Both directions are one kernel run twice: a banded matrix applied along the
// rows, the result stored transposed. Each thread holds one column and eight
// consecutive output rows, whose bands overlap, so an input value is loaded once
// for eight products; the weights come from a table of eight per input row
// (zeros outside a band), broadcast from shared memory. What bounds it: those
// shared-memory reads, three for eight products, and on small images the latency of
// the loads (a thread that summed four groups in turn left seven warps an SM; a
// thread a group: both applications at 2048 x 2048 66 -> 38 us, at 1100 34 -> 21).
#include "pc_internal.cuh"

namespace pc {
namespace {

constexpr int RS_COLS = 128;   // columns per CTA
constexpr int RS_ROWS = 32;    // output rows per CTA: four groups of eight
constexpr int RS_THREADS = RS_COLS * (RS_ROWS / 8);   // a column and a group each

// Band tables: group g of eight output rows starts at input row first[g] and
// holds `width` rows of eight weights. Up: output rows are the N pixels; down:
// the Nt small ones (the transpose), with the weights that the first one holds.
// Float64 arithmetic bounds it (2 operations a cycle and SM): a Horner
// sum instead of the series term by term with its divisions, and every weight
// once instead of twice: 146 -> 16 us for the tables at N = 1100, 314 us at 4096 before.
__global__ void k_band_up(const __grid_constant__ Taps t, int groups, int width, int* __restrict__ first,
                          float* __restrict__ w) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= groups * width * 8) return;
  const int r = e & 7, in = (e >> 3) % width, g = (e >> 3) / width;
  const int out = 8 * g + r, f = tap_first(t, 8 * g), k = f + in;
  if (r == 0 && in == 0) first[g] = f;
  double v = 0.0;
  if (out < t.N && k >= 0 && k < t.Nt) {
    const int k0 = tap_first(t, out);
    const double x = tap_x(t, out) - k;
    if (k >= k0 && k < k0 + t.K) v = tap_weight(t, x, sinpi(x));
  }
  w[e] = (float)v;
}

__global__ void k_band_down(const __grid_constant__ Taps t, int groups, int width, const int* __restrict__ up_first,
                            const float* __restrict__ up_w, int up_width, int* __restrict__ first,
                            float* __restrict__ w) {
  const int g = blockIdx.x;
  __shared__ int s_f;
  if (threadIdx.x == 0) {
    // first pixel whose taps reach row 8 g: tap_first(i) + K > 8 g
    int f = (int)ceil((8 * g - t.K / 2 - t.Nt / 2) * t.d) + t.N / 2 - 2;
    f = max(f, 0);
    while (f < t.N && tap_first(t, f) + t.K <= 8 * g) ++f;
    s_f = f;
    first[g] = f;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < width * 8; e += blockDim.x) {
    const int i = s_f + (e >> 3), k = 8 * g + (e & 7);
    float v = 0.f;
    if (k < t.Nt && i < t.N) {
      const int at = k - up_first[i >> 3];          // the up table holds zeros outside a band
      if (at >= 0 && at < up_width) v = up_w[((size_t)(i >> 3) * up_width + at) * 8 + (i & 7)];
    }
    w[(size_t)g * width * 8 + e] = v;
  }
}

// out[c][o] = scale * sum_t w[o][t] in[first + t][c]: in has n_in rows of n_cols,
// out n_cols rows of n_out (transposed). The last application of the adjoint
// also takes the maxima (maxbits, as the FFT epilogue).
__global__ void __launch_bounds__(RS_THREADS)
k_band_apply(const float* __restrict__ in, int n_in, int n_cols, const int* __restrict__ first,
             const float* __restrict__ w, int width, float* __restrict__ out, int n_out, float scale,
             unsigned* __restrict__ maxbits) {
  extern __shared__ float4 rs_w[];                         // 4 groups x width x 8 weights
  __shared__ float tile[RS_ROWS][RS_COLS + 1];
  const int tid = threadIdx.x, col = tid % RS_COLS, g = tid / RS_COLS;
  const int c0 = blockIdx.x * RS_COLS, o0 = blockIdx.y * RS_ROWS;
  const int c = min(c0 + col, n_cols - 1);
  const int groups = (n_out + 7) / 8, g0 = o0 / 8, gn = min(RS_ROWS / 8, groups - g0);
  const float4* src = reinterpret_cast<const float4*>(w) + (size_t)g0 * width * 2;
  for (int e = tid; e < gn * width * 2; e += RS_THREADS) rs_w[e] = src[e];
  __syncthreads();
  if (g < gn) {
    const int f = first[g0 + g];
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const float4* wg = rs_w + (size_t)g * width * 2;
#pragma unroll 8
    for (int t = 0; t < width; ++t) {
      const float v = in[(size_t)min(max(f + t, 0), n_in - 1) * n_cols + c];
      const float4 a = wg[2 * t], b = wg[2 * t + 1];
      acc[0] = fmaf(a.x, v, acc[0]);
      acc[1] = fmaf(a.y, v, acc[1]);
      acc[2] = fmaf(a.z, v, acc[2]);
      acc[3] = fmaf(a.w, v, acc[3]);
      acc[4] = fmaf(b.x, v, acc[4]);
      acc[5] = fmaf(b.y, v, acc[5]);
      acc[6] = fmaf(b.z, v, acc[6]);
      acc[7] = fmaf(b.w, v, acc[7]);
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) tile[8 * g + r][col] = acc[r] * scale;
  }
  __syncthreads();
  // 32 consecutive outputs of one column per warp
  const int lane = tid & 31, warp = tid >> 5, o = o0 + lane;
  float amax = 0.f;
  unsigned skey = 0;   // order-preserving key of the signed maximum (0 below every number)
  if (o < n_out) {
    for (int q = warp; q < RS_COLS && c0 + q < n_cols; q += RS_THREADS / 32) {
      const float m = tile[lane][q];
      out[(size_t)(c0 + q) * n_out + o] = m;
      amax = fmaxf(amax, fabsf(m));
      if (m != m) amax = __int_as_float(0x7fc00000);
      skey = max(skey, float_order_key(m));
    }
  }
  if (!maxbits) return;
  unsigned bits = __float_as_uint(amax);
  for (int off = 16; off; off >>= 1) {
    bits = max(bits, __shfl_xor_sync(0xffffffffu, bits, off));
    skey = max(skey, __shfl_xor_sync(0xffffffffu, skey, off));
  }
  if (lane == 0) {
    atomicMax(maxbits, bits);
    atomicMax(maxbits + 1, skey);
  }
}

int apply(const float* in, int n_in, int n_cols, const BandTable& t, float* out, int n_out, float scale,
          unsigned* maxbits, cudaStream_t st) {
  constexpr size_t row = (RS_ROWS / 8) * 8 * sizeof(float);   // of the table, four groups
  if (t.width > RS_MAX_WIDTH) return fail(PC_ERR_CAPACITY, "interpolation: a band of %d rows", t.width);
  const size_t smem = row * t.width;
  static bool attr = false;
  if (!attr) {
    PC_CUDA(cudaFuncSetAttribute(k_band_apply, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(row * RS_MAX_WIDTH)));
    attr = true;
  }
  k_band_apply<<<dim3(ceil_div(n_cols, RS_COLS), ceil_div(n_out, RS_ROWS)), RS_THREADS, smem, st>>>(
      in, n_in, n_cols, t.first, t.w, t.width, out, n_out, scale, maxbits);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

}  // namespace

int fill_band_tables(const Resample& r, int N, BandTable* up, BandTable* down, cudaStream_t st) {
  const Taps t = make_taps(r, N);
  const int gu = ceil_div(N, 8), gd = ceil_div(r.Nt, 8);
  k_band_up<<<ceil_div((int64_t)gu * up->width * 8, 128), 128, 0, st>>>(t, gu, up->width, up->first, up->w);
  k_band_down<<<gd, 128, 0, st>>>(t, gd, down->width, up->first, up->w, up->width, down->first, down->w);
  PC_LAUNCH_CHECK();
  return PC_OK;
}

// img (N x N) = scale * interpolation of the plan's small image
int launch_upsample(pc_plan_s* p, float* img, float scale, unsigned* maxbits, cudaStream_t st) {
  PC_TRY(apply(p->small_img, p->Nt, p->Nt, p->up, p->small_tmp, p->N, 1.0f, nullptr, st));
  return apply(p->small_tmp, p->Nt, p->N, p->up, img, p->N, scale, maxbits, st);
}

// the plan's small image = the transpose applied to img
int launch_downsample(pc_plan_s* p, const float* img, cudaStream_t st) {
  PC_TRY(apply(img, p->N, p->N, p->down, p->small_tmp, p->Nt, 1.0f, nullptr, st));
  return apply(p->small_tmp, p->N, p->Nt, p->down, p->small_img, p->Nt, 1.0f, nullptr, st);
}

}  // namespace pc
