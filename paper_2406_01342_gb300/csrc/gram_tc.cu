// Support contraction on the 5th-generation tensor cores (tcgen05):
//
//   G[a][c] = Re(Phi_A^H Phi_C)[a][c] = sum_k Re(Phi[k,a]) Re(Phi[k,c]) + Im(Phi[k,a]) Im(Phi[k,c])
//   b[a]    = Re(Phi_A^H V)[a]
//
// for the "new" atoms a (the MMA M dimension) against every active atom c and
// the visibility vector V (N), contracting over the visibilities (K: for each
// visibility its real and imaginary part, interleaved).
//
// Two kernels per K-chunk:
//  1. k_phase_gen evaluates every phase once -- exact fixed-point lattice turns
//     plus a double-float w-term, then sin/cos -- splits each value into
//     FP16 hi + lo and writes both into HBM in the exact K-major core-matrix
//     layout the tensor core reads (8 rows x 16 bytes per core matrix). Rows
//     are ordered as the caller gives the atoms (new atoms first), then one
//     row for V scaled by an exact power of two (so it fits FP16).
//  2. k_gram_bulk is a warp-specialised GEMM over tiles of 128 new atoms x up
//     to 256 columns: one producer thread streams the A and B rows of each 16-
//     visibility stage into a ring of shared-memory buffers with
//     cp.async.bulk (completion counted in bytes on an mbarrier); one thread
//     issues three tcgen05 MMAs per K-step (hi*hi + hi*lo + lo*hi, FP32
//     accumulate in tensor memory) and commits to the buffer's "empty"
//     mbarrier, which the producer waits on before refilling it; eight warps
//     drain the accumulators.
//
// Tiles. Symmetry gives the entries below the diagonal of the new atoms'
// block, so the columns of row tile i start at its own first row, 128 i, and
// are cut into equal chunks of at most 256 (a multiple of 16): about n^2 / 2 +
// 64 n products per visibility instead of the n^2 / 2 + 190 n of fixed 256-
// column tiles (874 rows: 439k against 622k). A chunk that starts on the
// diagonal holds the A rows too, which are then not copied a second time.
//
// Schedule (gram_sched.cuh). FP32 sums run over K-slices, float64 sums over the
// slices. A CTA takes one tile over a contiguous range of whole slices, the
// tiles of a range launched next to each other, so that the phase buffer is read
// from HBM once and then from L2.
//
// What binds it: shared-memory bandwidth. A stage of 256 columns takes 96 KB of
// operand reads and copies, 960 cycles at 128 B a cycle against the 768 of its
// MMAs (gb_stage_cycles). Measured, before (fixed 128 x 256 tiles, one CTA per
// K-slice, the drain between the MMAs) and after: 873 atoms x 200k visibilities
// 0.888 and 0.887 ms, 1001 x 1M 12.77 and 5.85 ms, 1602 x 200k 5.13 and 2.70 ms,
// 3000 x 200k 20.4 and 9.3 ms, 425 x 500k 0.92 and 0.76 ms; up to 1.16 PFLOP/s of
// distinct products (three FP16 products each).
//
// Accumulation: the tensor core adds each MMA result into its FP32 accumulator
// with truncation (measured: 2.6e-5 relative drift after ~750 adds). Each
// sub-slice of 256 visibilities (96 MMA adds per entry) therefore accumulates
// in one of two TMEM buffers, which the eight warps add, rounded to nearest,
// into FP32 registers (128 per thread) while the MMAs of the next sub-slice
// fill the other buffer; at the end of a slice they add the registers to a
// float64 accumulator in HBM.
//
// Every mbarrier wait is bounded (about 2 s of SM clock) and also watches a
// shared abort flag; on expiry the kernel sets *err, waits (bounded) for the
// copies and MMAs it issued, frees its tensor memory and returns, so the host
// reports PC_ERR_TIMEOUT instead of hanging the GPU.
#include <cuda_fp16.h>

#include "gram_sched.cuh"
#include "tcgen05.cuh"

namespace pc {
namespace {

constexpr int GB_KV = 16;               // visibilities per stage
constexpr int GB_ROW_BYTES = 4 * GB_KV; // 16 complex fp16 per row per stage = 64 bytes
constexpr int GB_KG = GB_KV / 4;        // 16-byte K-groups per row per stage
constexpr uint32_t GB_LBO = 128;        // K-adjacent core matrices
constexpr uint32_t GB_SBO = GB_KG * 128; // 8-row groups (512 bytes)
constexpr int GB_SMEM = 192 * 1024;     // stage buffers of a CTA: 4 of its widest tile's 48 KB,
constexpr int GB_NBUF = 12;             // more (at most this many) of a narrower one's
constexpr int GB_TLD = 33;              // row stride of a drain warp's 32 x 32 transpose (floats)
constexpr int GB_SMEM_ALL = GB_SMEM + 8 * 32 * GB_TLD * 4;
constexpr int GB_CHUNK = 8192;          // visibilities: granularity of a phase-buffer chunk
constexpr int GB_EPI = 256;             // warps 0-7 drain the accumulators
constexpr int GB_THREADS = GB_EPI + 64; // warp 8: producer, warp 9: MMA issue
constexpr long long GB_WAIT_CYCLES = 4000000000ll;

using tc::mma_commit;
using tc::mma_f16;
using tc::smem_u32;
using tc::tmem_ld32;

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) { return tc::smem_desc(saddr, GB_LBO, GB_SBO); }
__device__ __forceinline__ uint32_t instr_desc(int M, int N) { return tc::instr_desc_f16(M, N); }
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, volatile int* abort_flag) {
  return tc::mbar_wait(mbar, parity, abort_flag, GB_WAIT_CYCLES);
}

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// ------------------------------------------------------------------ phase generation

// max |Re V|, |Im V| over the visibilities (as float bits, non-negative floats order as uints).
__global__ void k_vmax(const float2* __restrict__ V, int64_t M, unsigned* __restrict__ bits) {
  float m = 0.f;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < M;
       k += (int64_t)gridDim.x * blockDim.x) {
    const float2 v = V[k];
    m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
  }
  for (int off = 16; off; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(bits, __float_as_uint(m));
}

// scale[0] = 2^-e, scale[1] = 2^e with 2^e > max component of V (exact powers of two).
__global__ void k_vscale(const unsigned* __restrict__ bits, float* __restrict__ scale) {
  const float m = __uint_as_float(*bits);
  int e = 0;
  if (m > 0.f && isfinite(m)) e = ilogbf(m) + 1;
  scale[0] = ldexpf(1.f, -e);
  scale[1] = ldexpf(1.f, e);
}

// One thread per (row, stage): the 16 visibilities of the stage for one atom
// (or the V row), as four 16-byte items of FP16 re/im pairs in hi and in lo.
// Item order equals memory order: [stage][row group][K-group][row in group],
// so a warp (32 consecutive rows) writes 4 x 128 contiguous bytes per K-group.
// The atom stays in registers across the stages a thread visits; every thread
// of a block visits the same stages, whose visibilities 16 threads copy into
// shared memory one stage ahead (asynchronous copies), so the phase work
// never waits on a global load.
// Threads 0..15 copy the visibilities of a stage into dst (asynchronously);
// every thread commits its (possibly empty) group of copies.
__device__ __forceinline__ void phase_prefetch(const int4* __restrict__ vis, int4* dst, int64_t k0, int64_t k_end,
                                               int stage, int n_stages) {
  if (threadIdx.x < GB_KV && stage < n_stages) {
    const int64_t k = k0 + (int64_t)stage * GB_KV + threadIdx.x;
    if (k < k_end) {
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst + threadIdx.x);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(vis + k) : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__global__ void __launch_bounds__(256, 6)
k_phase_gen(const int4* __restrict__ vis, const float2* __restrict__ V, int64_t k0, int64_t k_end,
            const float4* __restrict__ atoms, int n_atoms, int v_row, int rows_pad, int n_stages,
            const float* __restrict__ vscale, uint4* __restrict__ hi, uint4* __restrict__ lo) {
  __shared__ __align__(16) int4 s_vis[2][GB_KV];
  const int row = blockIdx.x * blockDim.x + threadIdx.x;
  const bool stored = row < rows_pad;                      // the last block may reach past the buffer
  const float sc = V ? vscale[0] : 0.f;
  const bool is_atom = row < n_atoms, is_v = row == v_row;
  const float4 at = is_atom ? atoms[row] : make_float4(0.f, 0.f, 0.f, 0.f);
  const size_t row_item = (size_t)(row >> 3) * (GB_KG * 8) + (row & 7);
  const size_t stage_items = (size_t)rows_pad * GB_KG;
  int b = 0;
  phase_prefetch(vis, s_vis[0], k0, k_end, blockIdx.y, n_stages);
  for (int stage = blockIdx.y; stage < n_stages; stage += gridDim.y, b ^= 1) {
    phase_prefetch(vis, s_vis[b ^ 1], k0, k_end, stage + gridDim.y, n_stages);
    asm volatile("cp.async.wait_group 1;" ::: "memory");   // this stage's copies landed
    __syncthreads();
    const int64_t kbase = k0 + (int64_t)stage * GB_KV;
    const size_t base = (size_t)stage * stage_items + row_item;
#pragma unroll
    for (int kg = 0; kg < GB_KG; ++kg) {
      uint32_t h[4], l[4];
#pragma unroll
      for (int v = 0; v < 4; v += 2) {
        float re[2], im[2];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const int j = kg * 4 + v + s;
          const int64_t k = kbase + j;
          re[s] = 0.f;
          im[s] = 0.f;
          if (k < k_end) {
            if (is_atom) {
              float sn, cs;
              __sincosf(6.283185307179586f * phase_turns(s_vis[b][j], at), &sn, &cs);
              re[s] = cs * at.w;
              im[s] = sn * at.w;
            } else if (is_v) {
              const float2 vv = V[k];
              re[s] = vv.x * sc;
              im[s] = -vv.y * sc;
            }
          }
        }
        // pairs (re, im) of two visibilities: split each into hi + lo
        tc::split_f16x2(re[0], im[0], h[v], l[v]);
        tc::split_f16x2(re[1], im[1], h[v + 1], l[v + 1]);
      }
      const size_t item = base + (size_t)kg * 8;
      if (stored) {
        hi[item] = make_uint4(h[0], h[1], h[2], h[3]);
        lo[item] = make_uint4(l[0], l[1], l[2], l[3]);
      }
    }
    __syncthreads();   // every read of s_vis[b] ended before the next prefetch overwrites it
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// ------------------------------------------------------------------ bulk-copy GEMM

struct GbArgs {
  const unsigned char* hi;   // phase buffer (this chunk)
  const unsigned char* lo;
  int rows_pad;
  int n_stages;              // stages in this chunk
  int nA;                    // rows of A (new atoms, the first rows)
  int nB;                    // columns: atoms + the V row
  int v_col;                 // column index of V, or -1
  const float* vscale;       // [1] = 2^e, multiplies the V column
  uint32_t tmem_cols;        // two accumulator buffers
  double* acc;
  int ldacc;
  int* err;
  int withhold;              // self-test: issue no MMA / commit, so the first buffer wait expires
  int tiles, slice, stages;  // GbPlan
};

__global__ void __launch_bounds__(GB_THREADS, 1) k_gram_bulk(const __grid_constant__ GbArgs g) {
  extern __shared__ __align__(1024) unsigned char gb_sm[];
  __shared__ __align__(8) uint64_t full_bar[GB_NBUF];
  __shared__ __align__(8) uint64_t empty_bar[GB_NBUF];
  __shared__ __align__(8) uint64_t tfull_bar[2], tempty_bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_abort;
  __shared__ int s_issued, s_consumed, s_last;   // stages copied / consumed, last committed

  const GbUnit u = gb_unit((int)blockIdx.x, g.tiles, g.stages, g.n_stages, g.nB);
  const int n = u.n, nst = u.count;
  const bool diag = u.a0 == u.b0;                     // the A rows are the chunk's first columns
  const int b_rows = diag ? max(n, GB_M) : n;
  const int a_bytes = diag ? 0 : GB_M * GB_ROW_BYTES; // 8 KB
  const int b_bytes = b_rows * GB_ROW_BYTES;
  const int buf_bytes = 2 * a_bytes + 2 * b_bytes;
  // in bytes, as much in flight for a narrow tile as for a wide one
  const int nbuf = min(GB_NBUF, GB_SMEM / buf_bytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const size_t stage_stride = (size_t)g.rows_pad * GB_ROW_BYTES;

  if (tid == 0) {
    for (int b = 0; b < GB_NBUF; ++b) {
      tc::mbar_init(smem_u32(&full_bar[b]), 1);
      tc::mbar_init(smem_u32(&empty_bar[b]), 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(smem_u32(&tfull_bar[b]), 1);
      tc::mbar_init(smem_u32(&tempty_bar[b]), GB_EPI / 32);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_abort = 0;
    s_issued = 0;
    s_consumed = 0;
    s_last = -1;
  }
  __syncwarp();
  if (warp == 0) tc::tmem_alloc(&tmem_slot, g.tmem_cols);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tmem_slot;
  const uint32_t half_cols = g.tmem_cols >> 1;

  if (warp == 8) {
    // ---------------- producer: one thread streams the stage tiles
    if (lane == 0) {
      int b = 0;
      uint32_t phase = 1;                            // of the buffer's "empty" barrier: its first use is free
      for (int i = 0; i < nst; ++i) {
        if (i >= nbuf && !mbar_wait(smem_u32(&empty_bar[b]), phase, &s_abort)) {
          s_abort = 1;
          break;
        }
        if (s_abort) break;
        const size_t soff = (size_t)(u.first + i) * stage_stride;
        unsigned char* dst = gb_sm + (size_t)b * buf_bytes;
        const uint32_t fb = smem_u32(&full_bar[b]);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"((uint32_t)buf_bytes)
                     : "memory");
        auto copy = [&](unsigned char* d, const unsigned char* src, uint32_t bytes) {
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                  smem_u32(d)),
              "l"(src), "r"(bytes), "r"(fb)
              : "memory");
        };
        if (!diag) {
          copy(dst, g.hi + soff + (size_t)u.a0 * GB_ROW_BYTES, (uint32_t)a_bytes);
          copy(dst + a_bytes, g.lo + soff + (size_t)u.a0 * GB_ROW_BYTES, (uint32_t)a_bytes);
        }
        copy(dst + 2 * a_bytes, g.hi + soff + (size_t)u.b0 * GB_ROW_BYTES, (uint32_t)b_bytes);
        copy(dst + 2 * a_bytes + b_bytes, g.lo + soff + (size_t)u.b0 * GB_ROW_BYTES, (uint32_t)b_bytes);
        s_issued = i + 1;
        if (++b == nbuf) {
          b = 0;
          phase ^= 1;
        }
      }
    }
    __syncwarp();
  } else if (warp == 9) {
    // ---------------- MMA issue: one thread
    if (lane == 0) {
      const uint32_t idesc = instr_desc(GB_M, n);
      int b = 0;
      uint32_t phase = 0;
      int in_slice = 0, sub = 0;                     // stage of the slice; sub-slices begun before
      for (int i = 0; i < nst; ++i) {
        const int tb = sub & 1;
        const bool first = in_slice % GB_SUB == 0;
        // a TMEM buffer's second and later uses wait for its drain
        bool good = !first || sub < 2 ||
                    mbar_wait(smem_u32(&tempty_bar[tb]), (uint32_t)(((sub >> 1) - 1) & 1), &s_abort);
        if (good) good = mbar_wait(smem_u32(&full_bar[b]), phase, &s_abort);
        if (!good) {
          s_abort = 1;
          break;
        }
        s_consumed = i + 1;
        const int buf = b;
        if (++b == nbuf) {
          b = 0;
          phase ^= 1;
        }
        if (g.withhold) continue;
        tc::fence_after_sync();
        const uint32_t base = smem_u32(gb_sm + (size_t)buf * buf_bytes);
        const uint32_t b_hi = base + 2 * a_bytes, b_lo = b_hi + b_bytes;
        const uint32_t a_hi = base, a_lo = base + (diag ? b_bytes : a_bytes);
        const uint32_t t_acc = tmem + tb * half_cols;
#pragma unroll
        for (int ks = 0; ks < GB_KG / 2; ++ks) {     // K = 16 fp16 elements per MMA
          const uint32_t koff = ks * 2 * GB_LBO;
          const uint32_t acc_on = !first || ks != 0;
          mma_f16(t_acc, smem_desc(a_hi + koff), smem_desc(b_hi + koff), idesc, acc_on);
          mma_f16(t_acc, smem_desc(a_hi + koff), smem_desc(b_lo + koff), idesc, 1u);
          mma_f16(t_acc, smem_desc(a_lo + koff), smem_desc(b_hi + koff), idesc, 1u);
        }
        mma_commit(smem_u32(&empty_bar[buf]));
        s_last = i;
        const bool slice_end = ++in_slice == g.slice || i == nst - 1;
        if (slice_end || in_slice % GB_SUB == 0) {
          mma_commit(smem_u32(&tfull_bar[tb]));
          ++sub;
        }
        if (slice_end) in_slice = 0;
      }
    }
    __syncwarp();
  } else {
    // ---------------- drain: warp w owns TMEM lanes 32 (w % 4) .. + 31 (its
    // rows) and columns 128 (w / 4) .. + 127 of both buffers
    const int q = warp & 3, h = warp >> 2;
    float* tr = reinterpret_cast<float*>(gb_sm + GB_SMEM) + warp * 32 * GB_TLD;
    const float vmul = g.vscale ? g.vscale[1] : 1.f;
    bool ok = true;
    int sub = 0;
    for (int s0 = 0; s0 < nst && ok; s0 += g.slice) {
      float sum[128];
#pragma unroll
      for (int j = 0; j < 128; ++j) sum[j] = 0.f;
      for (int left = min(g.slice, nst - s0); left > 0; left -= GB_SUB, ++sub) {
        const int tb = sub & 1;
        if (!mbar_wait(smem_u32(&tfull_bar[tb]), (uint32_t)((sub >> 1) & 1), &s_abort)) ok = false;
        if (!__all_sync(0xffffffffu, ok)) {
          s_abort = 1;
          ok = false;
          break;
        }
        tc::fence_after_sync();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (128 * h + 32 * c < n) {
            uint32_t f[32];
            tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + tb * half_cols + (uint32_t)(128 * h + 32 * c), f);
#pragma unroll
            for (int j = 0; j < 32; ++j) sum[32 * c + j] += __uint_as_float(f[j]);
          }
        }
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&tempty_bar[tb]));
      }
      if (!ok) break;
      // the slice's sums to float64, transposed so that lanes hold columns:
      // a warp's reductions fall on consecutive addresses
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (128 * h + 32 * c >= n) break;
#pragma unroll
        for (int j = 0; j < 32; ++j) tr[lane * GB_TLD + j] = sum[32 * c + j];
        __syncwarp();
        const int cl = 128 * h + 32 * c + lane, col = u.b0 + cl;
        const float scale = col == g.v_col ? vmul : 1.f;
        double* dst = g.acc + (size_t)(u.a0 + 32 * q) * g.ldacc + col;
        if (cl < n && col < g.nB) {
          // rows past the last new atom, and entries that symmetry gives, stay out
          int r_end = min(32, g.nA - u.a0 - 32 * q);
          if (col < g.nA) r_end = min(r_end, col - u.a0 - 32 * q + 1);
          for (int r = 0; r < r_end; ++r)
            atomicAdd(dst + (size_t)r * g.ldacc, (double)(tr[r * GB_TLD + lane] * scale));
        }
        __syncwarp();
      }
    }
  }
  // On abort every copy and MMA already issued must finish before the CTA
  // exits: bounded waits on the "full" phases of the stages copied but not
  // consumed, and on the last MMA commit.
  __syncthreads();
  if (s_abort && tid == 0) {
    volatile int no_abort = 0;
    for (int i = s_consumed; i < s_issued; ++i)
      mbar_wait(smem_u32(&full_bar[i % nbuf]), (uint32_t)((i / nbuf) & 1), &no_abort);
    if (s_last >= 0)
      mbar_wait(smem_u32(&empty_bar[s_last % nbuf]), (uint32_t)((s_last / nbuf) & 1), &no_abort);
    atomicExch(g.err, 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  __syncwarp();
  if (warp == 0) tc::tmem_dealloc(tmem, g.tmem_cols);
}

}  // namespace

// acc[r][c] += Re(Phi_A^H [Phi_atoms | V])[r][c] for the nA first rows of the
// atom list (A) against all n_atoms atoms plus, when V is given, the V column
// (index n_atoms), except entries c < r with c < nA (tiles wholly below the
// diagonal are skipped; they mirror computed ones). acc must be cleared by the caller. err_dev (int) is set to
// 1 if a bounded wait expired. pbuf is the phase buffer (grown here).
int launch_gram_tc(const int4* vis_fx, const float2* V, int64_t M, const float4* atoms, int n_atoms,
                   int nA, double* acc, int ldacc, int* err_dev, cudaStream_t st, bool withhold,
                   DevBuf& pbuf, float* vscale_dev, unsigned* vbits_dev) {
  if (M <= 0 || nA <= 0 || n_atoms <= 0) return PC_OK;
  const int rows = n_atoms + (V ? 1 : 0);
  // the phase buffer's rows: whole 16-row operand groups, and whole A tiles
  const int rows_pad = std::max(ceil_div(rows, 16) * 16, ceil_div(nA, GB_M) * GB_M);
  // chunk of visibilities: the phase buffer (hi + lo) stays within ~2 GB
  const int64_t per_vis = (int64_t)(ceil_div(rows, 256) * 256) * 8;
  int64_t KC = (2ll << 30) / per_vis;
  KC = std::max<int64_t>(GB_CHUNK, (KC / GB_CHUNK) * GB_CHUNK);
  const int64_t Mpad = ((M + GB_KV - 1) / GB_KV) * GB_KV;
  KC = std::min(KC, Mpad);
  const size_t half = (size_t)rows_pad * KC * 4;
  PC_TRY(pbuf.ensure(2 * half));
  uint4* hi = pbuf.as<uint4>();
  uint4* lo = reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(pbuf.p) + half);
  static bool attr_set = false;
  if (!attr_set) {
    PC_CUDA(cudaFuncSetAttribute(k_gram_bulk, cudaFuncAttributeMaxDynamicSharedMemorySize, GB_SMEM_ALL));
    attr_set = true;
  }
  // timed as two classes: the phase generation (HBM-bound; the V scale with
  // the first chunk) and the contraction
  for (int64_t k0 = 0; k0 < M; k0 += KC) {
    const int64_t kc = std::min(KC, M - k0);
    const int n_stages = (int)((kc + GB_KV - 1) / GB_KV);
    {
      ProfScope ps(PROF_PHASE_GEN, st);
      ps.kernels = 1;
      if (V && k0 == 0) {
        PC_CUDA(cudaMemsetAsync(vbits_dev, 0, sizeof(unsigned), st));
        k_vmax<<<(int)std::min<int64_t>(1024, ceil_div(M, 256)), 256, 0, st>>>(V, M, vbits_dev);
        k_vscale<<<1, 1, 0, st>>>(vbits_dev, vscale_dev);
        PC_LAUNCH_CHECK();
        ps.kernels += 2;
      }
      // ~16 resident 256-thread blocks per SM; each thread walks stages with stride gridDim.y
      const int bx = ceil_div(rows_pad, 256);
      const int by = (int)std::min<int64_t>(n_stages, std::max<int64_t>(1, (int64_t)152 * 16 / bx));
      k_phase_gen<<<dim3(bx, by), 256, 0, st>>>(vis_fx, V, k0, k0 + kc, atoms, n_atoms, V ? n_atoms : -1,
                                                rows_pad, n_stages, vscale_dev, hi, lo);
      PC_LAUNCH_CHECK();
    }
    static int n_sm = 0;
    if (n_sm == 0) {
      int dev = 0;
      cudaGetDevice(&dev);
      if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n_sm <= 0) n_sm = 152;
    }
    const GbPlan plan = gb_schedule(rows, nA, n_stages, n_sm);
    GbArgs a{reinterpret_cast<const unsigned char*>(hi), reinterpret_cast<const unsigned char*>(lo),
             rows_pad, n_stages, nA, rows, V ? n_atoms : -1, V ? vscale_dev : nullptr, 0, acc, ldacc,
             err_dev, withhold ? 1 : 0, plan.tiles, plan.slice, plan.stages};
    a.tmem_cols = plan.widest <= 128 ? 256 : 512;
    ProfScope pg(PROF_GRAM_TC, st);
    pg.kernels = 1;
    k_gram_bulk<<<plan.ctas, GB_THREADS, GB_SMEM_ALL, st>>>(a);
    PC_LAUNCH_CHECK();
  }
  return PC_OK;
}

}  // namespace pc
