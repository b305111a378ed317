// Direct Neumann solve by cosine transforms: plans, tables and launch interface
// (kernels in fct.cu). Internal to libgdgs.
#pragma once

#include "gdgs_internal.cuh"

namespace gdgs {

constexpr int kFctMaxCycles = 3;      // refinement cycles of a direct solve

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
  float *uhi, *ulo, *spec, *image;  // uhi, ulo: the first and second correction
  int tight;  // the second part goes to a grid too (fct_back_kernel)
  double cells, inv_cells, rtol2;
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

// The mean of rho in two parts: `hi`, the float nearest to the sum the divergence left (its
// FP32 partial sums are off by ~1e-8 of a mean that dominates the field), is known from the
// start and what the transforms work on is rho - hi; `lo`, the mean of that, is its lowest
// cosine coefficient, which the column passes leave in ctrl->rho_mean (the later ones what the
// rounding of the transform left of it, 1e-8 of the field's deviation).
__device__ __forceinline__ float fct_mean_hi(const Ctrl *ctrl, int c, double inv_cells) {
  return (float)(ctrl->rho_sum[c] * inv_cells);
}
// Where the first rows pass leaves sum (rho - hi)^2 (for rtol >= 1, where no pass but the finalize
// runs, that leaves ||rho - mean||^2), and the first rows-back pass the square of the residual
// that rtol asks for.
__host__ __device__ constexpr int fct_sq_slot(int c) { return fct_slot(kFctMaxCycles + 2, c); }
__host__ __device__ constexpr int fct_goal_slot(int c) { return fct_slot(kFctMaxCycles + 3, c); }

// By one thread of the first rows-back pass, which has the low part and `sq`: ||rho - mean||^2 (0
// where the difference is only the rounding of its two terms: a constant field) and the goal, so
// that the blocks of the later passes compare and do not compute in FP64 (0.7 us a launch).
__device__ __forceinline__ void fct_record_goal(const FctArgs &a, int c, float lo, double sq) {
  const double m2 = (double)lo * lo * a.cells, r0 = sq - m2, r = r0 > 1e-5 * m2 ? r0 : 0.0;
  a.ctrl->rnorm2[fct_slot(0, c)] = r;
  a.ctrl->rnorm2[fct_goal_slot(c)] = a.rtol2 * r;
}

// Whether channel c needs no further cycle after `k` cycles, and the number it has had
// (its residual after 1 .. k cycles is recorded, 0 cycles: a zero right-hand side). The
// rounding of the forward transforms is white noise of ~1e-7 of rho, which the division by
// lambda amplifies in the lowest modes (5e-5 of the image on 200 x 3 pixels at a relative
// residual of 4e-7), so the first cycle ends a solve only far below rtol.
__device__ __forceinline__ int fct_cycles_done(const Ctrl *ctrl, int c, int k, bool *done) {
  // all loads at once (each takes most of a microsecond, and every block waits for them)
  const double r0 = ctrl->rnorm2[fct_slot(0, c)], goal = ctrl->rnorm2[fct_goal_slot(c)];
  double r[kFctMaxCycles];
#pragma unroll
  for (int q = 1; q <= kFctMaxCycles; ++q) r[q - 1] = ctrl->rnorm2[fct_slot(q, c)];
  int n = k;
  *done = false;
#pragma unroll
  for (int q = kFctMaxCycles; q >= 1; --q)
    if (q <= k && r[q - 1] <= (q == 1 ? 1e-4 * goal : goal)) {
      *done = true;
      n = q;
    }
  if (r0 == 0.0) {
    *done = true;
    n = 0;
  }
  return n;
}
// Whether a pass has nothing to do in channel c: after `k` cycles, as above. k < 0: a pass of the
// first cycle, before the goal is known, which only a zero field (kFctRows) or one that is its
// mean (kFctFirst) can skip, or any for rtol >= 1; *sq is then the sum of squares it went by.
enum { kFctRows = -2, kFctFirst = -1 };
__device__ __forceinline__ bool fct_skip(const FctArgs &a, int c, int k, double *sq) {
  bool skip;
  if (k < 0) {
    *sq = *(k == kFctRows ? &a.ctrl->rho_sq[c] : &a.ctrl->rnorm2[fct_sq_slot(c)]);
    skip = (a.rtol2 >= 1.0) | (*sq == 0.0);
  } else {
    fct_cycles_done(a.ctrl, c, k, &skip);
  }
  return skip;
}
__device__ __forceinline__ bool fct_block_skip(const FctArgs &a, int c, int k) {
  __shared__ bool s_skip;
  double sq;
  if (threadIdx.x == 0) s_skip = fct_skip(a, c, k, &sq);
  __syncthreads();
  return s_skip;
}
// The same with the mean of the channel's rho.
struct FctChannel {
  float hi, lo;
  bool skip;
  double sq;  // (k < 0)
};
__device__ __forceinline__ FctChannel fct_block_channel(const FctArgs &a, int c, int k) {
  __shared__ FctChannel s_c;
  if (threadIdx.x == 0) {
    FctChannel f;
    f.hi = fct_mean_hi(a.ctrl, c, a.inv_cells);
    f.lo = a.ctrl->rho_mean[c];
    f.sq = 0.0;
    f.skip = fct_skip(a, c, k, &f.sq);
    s_c = f;
  }
  __syncthreads();
  return s_c;
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

// L u without rounding errors that matter, in plain FP32: the
// first correction u_1 is stored rounded to multiples of one power of two g per channel,
// about ulp(8 rms(u_1)) (fct_grid), so its differences and their sums are exact (below
// 2^24 g; beyond, they round relative to themselves), and rho - mean minus that sum loses nothing
// where the two cancel (FctResidual). u can be 1e5 times as large as L u (smooth right-hand sides,
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
// Where the sum of squares of the correction of cycle 0 and of cycle 1 goes.
__host__ __device__ constexpr int fct_grid_slot(int cycle, int c) {
  return fct_slot(kFctMaxCycles + (cycle ? 4 : 1), c);
}

// What is left of rho - mean after the exact sums L u of the iterate's parts, as an unevaluated
// sum hi + lo whose differences keep their rounding errors (Knuth's two-sum). The mean comes
// off first: next to a mean of 30 deviations, rho - L u would keep 5 bits fewer of the residual
// (images 1e-4 to 3e-2 of their range off, with a residual of exactly 0). And the residual after
// one part can exceed rho itself (smooth fields: six times at 4096 points), where rounding it to
// FP32 would leave 1e-7 of rho for good.
struct FctResidual {
  float hi, lo;
  __device__ __forceinline__ FctResidual(float rho, float mean_hi, float mean_lo) : hi(rho), lo(-mean_lo) { minus(mean_hi); }
  __device__ __forceinline__ void minus(float x) {
    const float t = __fsub_rn(hi, x), b = __fsub_rn(t, hi);
    lo = __fadd_rn(lo, __fsub_rn(__fsub_rn(hi, __fsub_rn(t, b)), __fadd_rn(x, b)));
    hi = t;
  }
  __device__ __forceinline__ float value() const { return __fadd_rn(hi, lo); }
};

}  // namespace gdgs
