// Direct Neumann solve (Eq. p2d) by cosine transforms, refined to the caller's rtol.
// Measured on a GB300 against the multigrid cycles it takes over from: 1920x1080x3 from
// maps 744 -> 207 us, 1355x757x3 (Bluestein) 780 -> 292 us, 3840x2160x1 1400 -> 270 us,
// 128x96x1 221 -> 55 us; relative error of the image 1.5e-6 -> 1e-7 (1080p).
//
// On the pixel grid the 5-point Neumann Laplacian is diagonal in the DCT-II modes of
// the two sides (Sec. 2.1 lists Fourier-type solvers beside multigrid): with
// lambda(ky, kx) = -4 sin^2(pi ky / 2H) - 4 sin^2(pi kx / 2W), e = IDCT(DCT(r) / lambda)
// solves L e = r exactly up to FP32 rounding. One cycle is three passes over the image:
//   rows      residual r of the current iterate, its DCT along x        -> spectrum
//   columns   DCT along y, the division by lambda, inverse DCT along y  -> spectrum
//   rows back inverse DCT along x: the correction e
// FP32 rounding of e leaves a relative residual of ~1e-5 (it is the size of the image's
// own FP32 representation error), and the next cycle solves for exactly that: the
// residual is evaluated without rounding errors that matter (fct_lap, FctResidual), so two
// cycles reach ~1e-7 or less, three 1e-9 (3e-8 where the field is the lowest mode of 3800 points). The multigrid needs 4-6 cycles, each a chain of ~12 dependent
// launches whose small levels leave the GPU idle (1080p, three channels: 150 us per
// cycle, all latency); here every launch covers all channels and every SM.
//
// A transform of n points works on two real sequences at once, packed as the real and
// imaginary part of one complex FFT of n points (Makhoul's even-odd order), held in
// shared memory. The FFT is mixed-radix Stockham, one radix-R butterfly set per thread
// in registers between two barriers, in place. Sides that are not in the list of
// fct_pass.cuh (83 even products of two or three radices up to 16 without 7, 11 and 13; no odd
// side, and not 448 = 64 * 7 or 2000 = 16 * 125) use Bluestein's chirp convolution on a
// length >= 2 n - 1 instead: two FFTs of that length per transform.
#include <stdlib.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "fct.cuh"

namespace gdgs {

const FctKernels *fct_slice0(int *);
const FctKernels *fct_slice1(int *);
const FctKernels *fct_slice2(int *);
const FctKernels *fct_slice3(int *);
const FctKernels *fct_slice4(int *);
const FctKernels *fct_slice5(int *);
const FctKernels *fct_slice6(int *);
const FctKernels *fct_slice7(int *);
const FctKernels *fct_slice8(int *);
const FctKernels *fct_slice9(int *);
const FctKernels *fct_slice10(int *);
const FctKernels *fct_slice11(int *);
const FctKernels *fct_slice12(int *);
const FctKernels *fct_slice13(int *);
const FctKernels *fct_slice14(int *);
const FctKernels *fct_slice15(int *);

namespace {

// After `k` cycles: image = u + (m_c - mean u) of the iterate channel c stopped at, and
// (when that is the k-th) its residual. Skipped when an earlier call already finished c.
// Third: the iterate has a third part (k = 3).
template <int V, bool Third>
__global__ void __launch_bounds__(256) fct_finalize_kernel(const __grid_constant__ FctArgs a, int k, int first) {
  griddep_enter();
  const int c = blockIdx.y;
  __shared__ int s_kf, s_skip;
  __shared__ float s_shift, s_hi, s_lo;
  if (threadIdx.x == 0) {
    bool done;
    const float hi = fct_mean_hi(a.ctrl, c, a.inv_cells), lo = a.ctrl->rho_mean[c];
    double su[kFctMaxCycles];  // sums of the corrections
#pragma unroll
    for (int q = 0; q < kFctMaxCycles; ++q) su[q] = a.ctrl->sum_u[q + 1][c];
    const int kf = fct_cycles_done(a.ctrl, c, k - 1, &done);
    s_skip = done && !first;
    s_kf = done ? kf : k;
    float mc = a.mean[0];
#pragma unroll
    for (int i = 1; i < GDGS_MAX_CHANNELS; ++i)
      if (i == c) mc = a.mean[i];
    double sum = 0.0;  // of u
#pragma unroll
    for (int q = 0; q < kFctMaxCycles; ++q)
      if (q < (done ? kf : k)) sum += su[q];
    s_shift = (float)((double)mc - sum * a.inv_cells);
    s_hi = hi;
    s_lo = lo;
    if (blockIdx.x == 0 && !s_skip) {
      a.ctrl->kf_c[c] = s_kf;
      a.ctrl->mean_set[c] = mc;
      if (a.rtol2 >= 1.0) {  // no pass ran that records it
        const double m = a.ctrl->rho_sum[c];
        a.ctrl->rnorm2[fct_sq_slot(c)] = fmax(a.ctrl->rho_sq[c] - m * m * a.inv_cells, 0.0);
      }
    }
  }
  __syncthreads();
  if (s_skip) return;
  const float hi = s_hi, lo = s_lo;
  const int kf = s_kf, W = a.W, H = a.H;
  const float shift = s_shift;
  const size_t plane = (size_t)H * W;
  const float *rho = a.rho + c * plane, *uh = a.uhi + c * plane, *ul = a.ulo + c * plane;
  float *img = a.image + c * plane;
  float r2 = 0.f;
  const int Wq = W / V, nq = H * Wq;  // H, W <= 4096
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x) {
    const int i = q / Wq, j0 = (q - i * Wq) * V, p = i * W + j0;
    if (kf == 0) {
#pragma unroll
      for (int d = 0; d < V; ++d) img[p + d] = 0.f + (0.f + shift);
      continue;
    }
    auto row = [&](const float *src, int o, float *dst) {
      if constexpr (V == 4) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(src + o));
        dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w;
      } else {
        dst[0] = __ldg(src + o);
      }
    };
    float r[V], h[V + 2], l[V + 2];
    row(rho, p, r);
#pragma unroll
    for (int d = 0; d < V; ++d) l[d + 1] = 0.f;
    // L of one part of the iterate
    auto lap = [&](const float *u, int pitch, float *c, float *out) {
      float s[V], n[V];
      const int o = i * pitch + j0;
      row(u, o, c + 1);
      row(u, i + 1 < H ? o + pitch : o, s);
      row(u, i > 0 ? o - pitch : o, n);
      c[0] = j0 > 0 ? __ldg(u + o - 1) : c[1];
      c[V + 1] = j0 + V < W ? __ldg(u + o + V) : c[V];
#pragma unroll
      for (int d = 0; d < V; ++d) out[d] = fct_lap(c[d + 1], c[d + 2], c[d], s[d], n[d]);
    };
    float lu[V], rl[V];
    lap(uh, W, h, lu);
#pragma unroll
    for (int d = 0; d < V; ++d) {
      FctResidual x(r[d], hi, lo);
      x.minus(lu[d]);
      r[d] = x.hi;
      rl[d] = x.lo;
    }
    if (kf > 1) {
      lap(ul, W, l, lu);
#pragma unroll
      for (int d = 0; d < V; ++d) r[d] -= lu[d];  // (what is left is about as large: nothing is lost)
    }
    if (Third && kf > 2) {
      float t[V + 2];
      lap(a.spec + (size_t)c * H * a.wp, a.wp, t, lu);
#pragma unroll
      for (int d = 0; d < V; ++d) {
        rl[d] -= lu[d];
        l[d + 1] += t[d + 1];
      }
    }
    float o[V];
#pragma unroll
    for (int d = 0; d < V; ++d) {
      r[d] += rl[d];
      r2 = fmaf(r[d], r[d], r2);
      o[d] = h[d + 1] + (l[d + 1] + shift);
    }
    if constexpr (V == 4) *reinterpret_cast<float4 *>(img + p) = make_float4(o[0], o[1], o[2], o[3]);
    else img[p] = o[0];
  }
  r2 = fct_block_sum(r2);
  if (threadIdx.x == 0 && kf == k) atomicAdd(&a.ctrl->rnorm2[fct_slot(k, c)], (double)r2);
}

// ------------------------------------------------------------------ plans (host)

// Every FFT length, ascending, the direct ones before the Bluestein ones.
const std::vector<FctKernels> &lengths() {
  static const std::vector<FctKernels> all = [] {
    const FctKernels *(*slices[kFctSlices])(int *) = {fct_slice0, fct_slice1, fct_slice2, fct_slice3, fct_slice4, fct_slice5, fct_slice6, fct_slice7, fct_slice8, fct_slice9, fct_slice10, fct_slice11, fct_slice12, fct_slice13, fct_slice14, fct_slice15};
    std::vector<FctKernels> v;
    for (auto s : slices) {
      int n = 0;
      const FctKernels *e = s(&n);
      v.insert(v.end(), e, e + n);
    }
    std::sort(v.begin(), v.end(), [](const FctKernels &a, const FctKernels &b) {
      return a.e.bluestein != b.e.bluestein ? a.e.bluestein < b.e.bluestein : a.e.len < b.e.len;
    });
    return v;
  }();
  return all;
}

// The FFT of one side: of n points if there is one, else the shortest that holds the
// chirp convolution; null above the longest.
const FctKernels *plan_side(int n, FctSide *d) {
  d->n = n;
  for (const FctKernels &k : lengths())
    if (k.e.bluestein ? k.e.len >= 2 * n - 1 : k.e.len == n) {
      d->bluestein = k.e.bluestein;
      d->len = k.e.len;
      return &k;
    }
  return nullptr;
}

size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

// GDGS_DIRECT=0 keeps the multigrid cycles; so do the switches of the multigrid's
// streaming passes (comparisons and tests name them).
bool fct_enabled() {
  static const bool on = [] {
    const char *v = getenv("GDGS_DIRECT");
    if (v) return v[0] != '0';
    return !getenv("GDGS_STREAM") && !getenv("GDGS_STREAM_ROWS") && !getenv("GDGS_STREAM_UP_LEVELS") &&
           !getenv("GDGS_STREAM_DOWN_LEVELS");
  }();
  return on;
}

// Opt the kernels of a length in to the shared memory their blocks take, once per device.
cudaError_t opt_in(const FctKernels &k) {
  static std::atomic<unsigned long long> done[160];
  int dev = 0;
  cudaError_t r = cudaGetDevice(&dev);
  if (r != cudaSuccess) return r;
  const size_t i = (size_t)(&k - lengths().data());
  const unsigned long long bit = 1ull << (dev & 63);
  if (i < 160 && (done[i].load(std::memory_order_acquire) & bit)) return cudaSuccess;
  const std::pair<FctKernel, int> need[4] = {
      {k.rows, k.e.row_smem}, {k.cols, k.e.col_smem}, {k.back, k.e.row_smem}, {k.chirp, k.e.chirp_smem}};
  // whatever the size: the kernels' static shared memory counts towards the 48 KB as well
  for (const auto &n : need)
    if (n.first && r == cudaSuccess)
      r = cudaFuncSetAttribute((const void *)n.first, cudaFuncAttributeMaxDynamicSharedMemorySize, n.second);
  if (r == cudaSuccess && i < 160) done[i].fetch_or(bit, std::memory_order_acq_rel);
  return r;
}

}  // namespace

// The direct solve takes every number of sweeps with the default relaxation and coarsest
// grid: a caller who sets one of these two gets the multigrid cycles he describes (all of
// them change the way to the solution, not the solution; with 1 + 1 sweeps the multigrid
// took 1084 us for 1617x768x4, the direct solve 337 us). Sides up to the longest FFT length, 4096
// points (Bluestein's convolution of 8192 points included).
bool fct_plan(const PoissonArgs &a, FctPlan *f) {
  if (a.omega != 1.2f || a.coarse_max_dim != 8 || !fct_enabled()) return false;
  if (a.H < 2 || a.W < 2) return false;
  f->ex = plan_side(a.W, &f->x);
  f->ey = plan_side(a.H, &f->y);
  if (!f->ex || !f->ey) return false;
  // Bluestein transforms cost two to three times a direct length, 0.10 ns a pixel and channel
  // with both sides, 0.067 with one; the multigrid, whose finest passes stream at even widths,
  // about 400 us + 0.05 ns. Large images of such sides keep it: 2176x2061x3 1423 (direct) and
  // 1125 us, x1 520 and 728; 3840x2153x3 1656 and 1614, 2560x2153x3 1167 and 1247; at odd
  // widths the direct solve is faster throughout (3833x2153x3 2442 and 3108).
  const int chirps = f->x.bluestein + f->y.bluestein;
  const long long work = (long long)a.H * a.W * a.C;
  if (a.W % 2 == 0 && ((chirps == 2 && work > 8000000) || (chirps == 1 && work > 22000000))) return false;
  f->cycles = std::min(a.max_cycles, kFctMaxCycles);
  f->wp = (a.W + 7) & ~7;
  // the arrays of the multigrid corrections and residuals, which this path does not use
  const Plan &p = *a.plan;
  size_t o = p.off_e0;
  f->spec = (float *)(a.ws + o);
  o = up256(o + sizeof(float) * (size_t)a.C * a.H * f->wp);
  FctSide *sides[2] = {&f->x, &f->y};
  for (FctSide *d : sides) {
    d->tw = (float2 *)(a.ws + o);
    o = up256(o + sizeof(float2) * (size_t)d->len);
    d->th = (float2 *)(a.ws + o);
    o = up256(o + sizeof(float2) * (size_t)d->n);
    d->s2 = (float *)(a.ws + o);
    o = up256(o + sizeof(float) * (size_t)d->n);
    if (d->bluestein) {
      d->chirp = (float2 *)(a.ws + o);
      o = up256(o + sizeof(float2) * (size_t)d->n);
      d->bhat = (float2 *)(a.ws + o);
      o = up256(o + sizeof(float2) * (size_t)d->len);
    }
  }
  return o <= p.total;
}

cudaError_t run_fct(const PoissonArgs &a, const FctPlan &f, const float *rho, float *uhi, float *ulo,
                    cudaStream_t st) {
  FctArgs fa{};
  fa.x = f.x;
  fa.y = f.y;
  fa.C = a.C;
  fa.H = a.H;
  fa.W = a.W;
  fa.wp = f.wp;
  fa.rho = rho;
  fa.uhi = uhi;
  fa.ulo = ulo;
  fa.tight = a.rtol < 1e-6f;
  fa.spec = f.spec;
  fa.image = a.image;
  fa.cells = (double)a.H * a.W;
  fa.inv_cells = 1.0 / fa.cells;
  fa.rtol2 = (double)a.rtol * a.rtol;
  for (int c = 0; c < GDGS_MAX_CHANNELS; ++c) fa.mean[c] = a.mean[c];
  fa.ctrl = a.ctrl;
  cudaError_t e = opt_in(*f.ex);
  if (e == cudaSuccess) e = opt_in(*f.ey);
  if (e != cudaSuccess) return e;
  const FctEntry &ex = f.ex->e, &ey = f.ey->e;
  for (int i = 0; i < 2; ++i) {
    const FctKernels &k = i ? *f.ey : *f.ex;
    if (!k.e.bluestein) continue;
    LaunchScope ls_("fct_chirp", st);
    launch_k(k.chirp, 1, k.e.chirp_threads, k.e.chirp_smem, st, fa, i);
  }
  const dim3 rg(((a.H + 1) / 2 + ex.row_g - 1) / ex.row_g, a.C), cg(((a.W + 1) / 2 + ey.col_g - 1) / ey.col_g, a.C);
  const int V = a.W % 4 == 0 ? 4 : 1;
  const long long nq = (long long)a.H * (a.W / V);
  const dim3 fg((unsigned)std::max<long long>(1, std::min<long long>((nq + 255) / 256, 608)), a.C);
  // The profile's names of a cycle's residual side and correction side on the finest grid are those of
  // the multigrid: callers find them there with either solver, and fct_columns tells which one ran.
  for (int k = 0; k < f.cycles; ++k) {
    {
      LaunchScope ls_("mg0_down", st);
      launch_k(f.ex->rows, rg, ex.row_threads, ex.row_smem, st, fa, k);
    }
    {
      LaunchScope ls_("fct_columns", st);
      launch_k(f.ey->cols, cg, ey.col_threads, ey.col_smem, st, fa, k);
    }
    {
      LaunchScope ls_("mg0_up", st);
      launch_k(f.ex->back, rg, ex.row_threads, ex.row_smem, st, fa, k);
    }
    if (k > 0 || f.cycles == 1) {
      const int first = k == std::min(1, f.cycles - 1);
      LaunchScope ls_("finalize", st);
      const auto fin = V == 4 ? (k > 1 ? fct_finalize_kernel<4, true> : fct_finalize_kernel<4, false>)
                              : (k > 1 ? fct_finalize_kernel<1, true> : fct_finalize_kernel<1, false>);
      launch_k(fin, fg, 256, 0, st, fa, k + 1, first);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace gdgs
