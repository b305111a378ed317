// Direct Neumann solve by cosine transforms: plans, tables and launch interface
// (kernels in fct.cu). Internal to libgdgs.
#pragma once

#include "gdgs_internal.cuh"

namespace gdgs {

constexpr int kFctMaxCycles = 3;      // refinement cycles of a direct solve
constexpr int kFctMaxThreads = 768;

// The transform of one side of the image: length n of the cosine transform, done by
// complex FFTs of `len` points: len == n when the library has an FFT of that length,
// else Bluestein's chirp convolution (len >= 2 n - 1).
struct FctSide {
  int n, len, bluestein;
  float2 *tw;     // [len]  exp(-2 pi i t / len)
  float2 *th;     // [n]    (cos, sin)(pi k / 2n)
  float *s2;      // [n]    4 sin^2(pi k / 2n)
  float2 *chirp;  // [n]    exp(-i pi t^2 / n)            (Bluestein)
  float2 *bhat;   // [len]  FFT of the conjugate chirp     (Bluestein)
};

// Arguments of the passes (fct_pass.cuh).
struct FctArgs {
  FctSide x, y;
  int C, H, W, wp;
  const float *rho;
  float *uhi, *ulo, *spec, *image;
  double inv_cells;
  float mean[GDGS_MAX_CHANNELS];
  Ctrl *ctrl;
};

// An FFT length: threads, transforms and shared-memory bytes of a block of its row and
// column kernels (and of the chirp kernel), and the kernels.
struct FctEntry {
  int len, bluestein;
  int row_threads, row_g, row_smem;
  int col_threads, col_g, col_smem;
  int chirp_threads, chirp_smem;
};
using FctKernel = void (*)(const FctArgs, int);
struct FctKernels {
  FctEntry e;
  FctKernel rows, cols, back, chirp;
};
constexpr int kFctSlices = 16;  // translation units the lengths are spread over

struct FctPlan {
  FctSide x, y;
  const FctKernels *ex, *ey;
  int cycles;        // refinement cycles launched
  int wp;            // row pitch of the spectrum (a multiple of 8 floats)
  float *spec;       // [C][H][wp]
};

// Whether the direct solve takes this problem, and its plan (tables and spectrum in
// the workspace arrays that only the multigrid cycles use).
bool fct_plan(const PoissonArgs &a, FctPlan *f);

// Everything after the divergence (which also fills the tables).
cudaError_t run_fct(const PoissonArgs &a, const FctPlan &f, const float *rho, float *uhi, float *ulo,
                    cudaStream_t st);

// (cos, sin)(2 pi t / n), 0 <= t < n: quarter turns are split off in integers, so the
// remaining angle is at most pi / 4 and its rounding no more than half an ulp of it.
__device__ __forceinline__ float2 fct_turn(int t, int n) {
  const int q = (4 * t + n / 2) / n;  // nearest quarter
  const float x = 0.5f * (float)(4 * t - q * n) / (float)n;  // half turns, |x| <= 1/4
  float s, c;
  sincospif(x, &s, &c);
  switch ((int)(q & 3)) {
    case 0: return make_float2(c, s);
    case 1: return make_float2(-s, c);
    case 2: return make_float2(-c, -s);
    default: return make_float2(s, -c);
  }
}

// The tables of one side, spread over `threads` threads.
__device__ __forceinline__ void fct_build_tables(const FctSide &d, int tid, int threads) {
  for (int i = tid; i < d.len; i += threads) {
    const float2 w = fct_turn(i, d.len);
    d.tw[i] = make_float2(w.x, -w.y);
  }
  for (int k = tid; k < d.n; k += threads) {
    d.th[k] = fct_turn(k, 4 * d.n);
    const float s = sinpif(0.5f * (float)k / (float)d.n);
    d.s2[k] = 4.f * s * s;
    if (d.bluestein) {
      const float2 w = fct_turn((k * k) % (2 * d.n), 2 * d.n);
      d.chirp[k] = make_float2(w.x, -w.y);
    }
  }
}

// ||rho - mean||^2 of channel c, and whether it needs no further cycle after `k` cycles
// (its residual after 1 .. k cycles is recorded, 0 cycles: a zero right-hand side). The
// rounding of the forward transforms is white noise of ~1e-7 of rho, which the division by
// lambda amplifies in the lowest modes (5e-5 of the image on 200 x 3 pixels at a relative
// residual of 4e-7), so the first cycle ends a solve only far below rtol.
__device__ __forceinline__ double fct_r0(const Ctrl *ctrl, int c, double inv_cells) {
  const double s = ctrl->rho_sum[c];
  return fmax(ctrl->rho_sq[c] - s * s * inv_cells, 0.0);
}
__device__ __forceinline__ int fct_cycles_done(const Ctrl *ctrl, int c, double inv_cells, int k, bool *done) {
  const double thr = ctrl->rtol * ctrl->rtol * fct_r0(ctrl, c, inv_cells);
  if (ctrl->rtol * ctrl->rtol >= 1.0 || fct_r0(ctrl, c, inv_cells) == 0.0) {
    *done = true;
    return 0;
  }
  for (int q = 1; q <= k; ++q)
    if (ctrl->rnorm2[fct_slot(q, c)] <= (q == 1 ? 1e-4 * thr : thr)) {
      *done = true;
      return q;
    }
  *done = false;
  return k;
}
__device__ __forceinline__ bool fct_block_done(const FctArgs &a, int c, int k) {
  __shared__ int s_done;
  if (threadIdx.x == 0) {
    bool d;
    fct_cycles_done(a.ctrl, c, a.inv_cells, k, &d);
    s_done = d;
  }
  __syncthreads();
  return s_done != 0;
}

// Block-wide sum; the result is valid in thread 0.
__device__ __forceinline__ float fct_block_sum(float v) {
  __shared__ float part[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.f;
  if (threadIdx.x == 0)
    for (int i = 0; i < (int)(blockDim.x + 31) / 32; ++i) s += part[i];
  return s;
}

// The residual rho - mean - L u without rounding errors that matter, in plain FP32: the
// first correction u_1 is stored rounded to multiples of one power of two g per channel,
// about ulp(8 rms(u_1)) (fct_grid), so its differences and their sums are exact (below
// 2^24 g; beyond, they round relative to themselves), and rho minus that sum loses nothing
// where the two cancel. u can be 1e5 times as large as L u (smooth right-hand sides,
// images spanning hundreds); with u_1 rounded to each value's own ulp the same sums were
// off by more than the 1e-6 of rho that a cycle has to see, and error-free transformations
// cost 70 instructions a pixel. The rounding itself is ~1e-6 of rms(u_1), like that of the
// transforms, and goes into the next correction.
__device__ __forceinline__ float fct_lap(float c, float e, float w, float s, float n) {
  return __fadd_rn(__fadd_rn(__fsub_rn(e, c), __fsub_rn(w, c)), __fadd_rn(__fsub_rn(s, c), __fsub_rn(n, c)));
}

// 3/2 2^23 g: adding and subtracting it rounds to multiples of g. sum2: the sum of squares
// of u_1's scaled cosine coefficients, at most 4 of which make up the mean square of u_1.
__device__ __forceinline__ float fct_grid(double sum2) {
  const float rms8 = 16.f * sqrtf((float)sum2);
  if (!(rms8 > 0.f) || !(rms8 < 1e37f)) return 0.f;
  return 3.f * exp2f(ceilf(log2f(rms8)));
}
__host__ __device__ constexpr int fct_grid_slot(int c) { return fct_slot(kFctMaxCycles + 1, c); }

// The mean of rho over channel c.
__device__ __forceinline__ float fct_block_mean(const FctArgs &a, int c) {
  __shared__ float s_m;
  if (threadIdx.x == 0) s_m = (float)(a.ctrl->rho_sum[c] * a.inv_cells);
  __syncthreads();
  return s_m;
}

}  // namespace gdgs
