// Backward of the render path: d(loss)/d(image) -> d(loss)/d(Gaussian parameters).
//
// The render is image = S(T(D(M(theta)))): M the front-to-back composite of the
// projected splats (Eq. gdgs2d), D the divergence (gradient attribute) or the
// identity (Laplacian attribute, Eq. gdgs), T the hard threshold (Eq. thresh),
// S the Neumann solve with the mean of rho removed and the supplied mean added
// (Eq. p2d). Backwards:
//   S^T  L is symmetric on zero-mean fields, so d rho = the same zero-mean solve
//        of d image (run by the caller's solver call into a second workspace);
//   T^T  d rho_raw = d rho where the threshold kept rho (rho != 0), else 0;
//   D^T  the transpose of the zero-flux divergence: d gx(i,j) = d rho(i,j) -
//        d rho(i,j+1) for j < W-1 (a negative forward difference), same for gy;
//        tiles the forward masked contribute nothing;
//   M^T  per tile, every pixel recomputes its forward pass (final transmittance
//        and last splat visited), then walks its splats back to front keeping
//        the transmittance before each splat (T / (1 - a)) and the attribute
//        composited behind it (B <- c a + (1 - a) B): dM/dc = a T_before,
//        dM/da = T_before (c - B); a = min(alpha_max, opacity 2^-p) gives the
//        opacity, centre and conic terms. Per-splat sums over a warp's pixels
//        go to global memory with atomics;
//   projection^T per Gaussian, from (d centre, d conic, d opacity) through
//        conic = Sigma2D^-1, Sigma2D = T Sigma T^T + dil I, T = J(t) W,
//        t = W mu + w, Sigma = R(q) S S^T R(q)^T and the quaternion's
//        normalisation. Alpha-test, stop and cull decisions have zero derivative.
#include <math.h>

#include "gdgs_internal.cuh"

namespace gdgs {

namespace {

__device__ __forceinline__ bool on_tile(const uint8_t *mask, int tiles_x, int i, int j) {
  return !mask || mask[(i / kTile) * tiles_x + (j / kTile)];
}

__global__ void __launch_bounds__(256) divergence_adjoint_kernel(DivAdjArgs a) {
  griddep_enter();
  const size_t plane = (size_t)a.H * a.W;
  const size_t total = plane * a.C;
  for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < total;
       p += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(p / plane);
    const size_t q = p - (size_t)c * plane;
    const int i = (int)(q / a.W), j = (int)(q - (size_t)i * a.W);
    const float *rb = a.rbar + (size_t)c * plane;
    const float *rf = a.rho_fwd ? a.rho_fwd + (size_t)c * plane : nullptr;
    auto r = [&](size_t o) { return (rf && rf[o] == 0.f) ? 0.f : rb[o]; };
    const bool on = on_tile(a.mask, a.tiles_x, i, j);
    if (a.input_is_rho) {
      a.mbar[(size_t)c * plane + q] = on ? r(q) : 0.f;
    } else {
      const float r0 = r(q);
      a.mbar[(size_t)(2 * c) * plane + q] = (on && j + 1 < a.W) ? r0 - r(q + 1) : 0.f;
      a.mbar[(size_t)(2 * c + 1) * plane + q] = (on && i + 1 < a.H) ? r0 - r(q + a.W) : 0.f;
    }
  }
}

// Sums N values over the warp's lanes, transposed: at every step a lane keeps half of its
// values and hands the other half to its partner, so N - 1 + log2(32 / N) shuffles give every
// sum to a lane of its own (13 for N = 12; a butterfly per value takes 60). Returns the sum
// and in *idx which one; idx >= N or an odd lane: nothing.
template <int N, int O>
__device__ __forceinline__ float warp_sums(float (&v)[N], int lane, int base, int *idx) {
  if constexpr (O == 0) {
    *idx = base;
    return v[0];
  } else {
    constexpr int H = (N + 1) / 2;
    const bool up = lane & O;
    float w[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const float hi = i + H < N ? v[i + H] : 0.f;
      if constexpr (N == 1) {
        w[i] = v[i] + __shfl_xor_sync(0xffffffffu, v[i], O);
      } else {
        w[i] = (up ? hi : v[i]) + __shfl_xor_sync(0xffffffffu, up ? v[i] : hi, O);
      }
    }
    if (N > 1 && up) base += H;
    // slots beyond this half's count hold zeros: an index past the half's end is void
    return warp_sums<H, O / 2>(w, lane, base, idx);
  }
}
// Which lanes hold a real sum: the index must lie in its half at every step.
template <int N, int O>
__device__ __forceinline__ bool warp_sums_valid(int lane, int count) {
  if constexpr (O == 0) {
    return count > 0;
  } else {
    constexpr int H = (N + 1) / 2;
    if constexpr (N == 1) {
      return !(lane & O) && warp_sums_valid<1, O / 2>(lane, count);
    } else {
      return warp_sums_valid<H, O / 2>(lane, (lane & O) ? max(0, count - H) : min(count, H));
    }
  }
}

// a / b of both elements: Newton-Raphson on an approximate reciprocal and Markstein's correction
// of the quotient by its exact remainder (IBM J. Res. Dev. 34, 1990). CUDA's own quotient, bit for
// bit, for a transmittance a of 1 to 2^-100 and b = 1 - alpha of 1 to 2^-24 (any alpha_max below
// 1; 2 10^9 samples); from about 2^-107 down the remainder underflows and an ulp may be lost.
__device__ __forceinline__ f32x2 div2(f32x2 a, f32x2 b) {
  float b0, b1, r0, r1;
  unpk(b, b0, b1);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(b0));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(b1));
  const f32x2 nb = mul2(b, pk(-1.f, -1.f));
  f32x2 r = pk(r0, r1);
  r = fma2(r, fma2(nb, r, pk(1.f, 1.f)), r);
  const f32x2 q = mul2(a, r);
  return fma2(fma2(nb, q, a), r, q);
}

// A float as a double by its bits (a conversion instruction runs on the FP64 pipe, which
// takes 16 cycles a warp here); subnormals become 0.
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
  if (e == 0x7f800000u) return (double)x;  // infinity, NaN
  const int hi = (int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u));
  return e == 0u ? 0.0 : __hiloint2double(hi, (int)(u << 29));
}

// Backward of the composite. As in the forward rasteriser a warp holds an 8 x 8 block of
// the tile, a lane two pixels of a column as packed pairs, and walks the tile's list on
// its own, 32 splats at a time: first front to back for the pixels' transmittances and
// last splats, then back to front. A splat's 6 + Q sums over the block's 64 pixels go to
// global memory in two coalesced atomic instructions; the six projected quantities are
// accumulated in FP64, because a splat can collect thousands of partial sums that nearly
// cancel (in FP32 the order of the atomics alone moved d quat by 3e-5). The second moments
// are those of w = 2 k2 conic d, not of the offsets d: Sigma2D's gradient -C (sum g d d^T) C is
// then a plain multiple of them, while through the moments of d an elongated splat's
// gradient is what remains of sums (length / width)^2 times as large.
// Measured on a GB300, 1280x720 with 500k Gaussians, three channels, the kernel alone: 1380
// (a pixel per lane, 60 shuffles and 12 single-lane atomics per splat and warp) -> 845 us; bound by
// issue (470M warp-instructions, 61 % issue active).
constexpr int kBwdThreads = 128;

template <int Q>
__global__ void __launch_bounds__(kBwdThreads, Q <= 6 ? 6 : 4) raster_backward_kernel(RasterBwdArgs a) {
  griddep_enter();
  constexpr int QP = (Q + 1) / 2;
  // per warp, up to 32 splats: store_pairs(), (-l_x, -l_y) and the attribute, all twice
  __shared__ float4 s_splat[kBwdThreads / 32][5 + QP][32];
  __shared__ float s_iopa[kBwdThreads / 32][32];  // 1 / opacity
  __shared__ uint32_t s_id[kBwdThreads / 32][32];
  __shared__ int s_pos[kBwdThreads / 32][32];     // place in the tile's list
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned ntiles = a.ctrl->n_active;
  if (blockIdx.x >= ntiles || a.ctrl->gave_up) return;  // no sorted list
  const int tile = (int)a.active[blockIdx.x];
  const int tyi = tile / a.tiles_x, txi = tile - tyi * a.tiles_x;
  const int x0 = txi * kTile, y0 = tyi * kTile;
  const int bx = 8 * (warp & 1), by = 8 * (warp >> 1);
  const int lx = bx + (lane & 7), ly = by + (lane >> 3);
  const int px = x0 + lx, py = y0 + ly;
  const bool in0 = px < a.W && py < a.H, in1 = px < a.W && py + 4 < a.H;
  const f32x2 fpx = pk(lx + 0.5f, lx + 0.5f), fpy = pk(ly + 0.5f, ly + 4.5f);
  const float x0f = (float)x0, y0f = (float)y0;
  const uint2 rg = tile_range(a.range, tile);
  const float amin = a.alpha_min, amax = a.alpha_max, tmin = a.t_min;
  const f32x2 minus1 = pk(-1.f, -1.f);
  float4(*S)[32] = s_splat[warp];

  // the splats of [s, s + 32) that reach the block, packed in list order; their number
  auto stage = [&](unsigned s, bool full) -> int {
    const unsigned j = s + lane;
    StagedSplat st;
    float4 kc;
    uint32_t g = 0;
    bool in = false;
    if (j < rg.y) {
      g = a.pval[j];
      kc = a.sconic[g];
      st = stage_splat(a.smean[g], kc, x0f, y0f);
      in = reaches_block<8>(st, kc, amin, by, bx);
    }
    const unsigned ball = __ballot_sync(0xffffffffu, in);
    __syncwarp();
    if (in) {
      const int k = __popc(ball & ((1u << lane) - 1u));
      store_pairs(st, &S[0][k], 32);
      s_pos[warp][k] = (int)j;
      if (full) {
        S[4][k] = make_float4(-st.lx, -st.lx, -st.ly, -st.ly);
        s_iopa[warp][k] = 1.f / kc.w;
        s_id[warp][k] = g;
        float gv[2 * QP];
        gv[2 * QP - 1] = 0.f;
#pragma unroll
        for (int q = 0; q < Q; ++q) gv[q] = __ldg(a.attr + (size_t)g * Q + q);
#pragma unroll
        for (int v = 0; v < QP; ++v) S[5 + v][k] = make_float4(gv[2 * v], gv[2 * v], gv[2 * v + 1], gv[2 * v + 1]);
      }
    }
    __syncwarp();
    return __popc(ball);
  };

  // 1. the forward pass again: final transmittances and the last splats composited
  float T0 = 1.f, T1 = 1.f;
  int last0 = -1, last1 = -1;
  bool live0 = in0, live1 = in1;
  for (unsigned s = rg.x; s < rg.y; s += 32) {
    if (!__any_sync(0xffffffffu, live0 || live1)) break;
    const int n = stage(s, false);
    for (int k = 0; k < n; ++k) {
      f32x2 X, Y;
      float t0, t1;
      staged_log2_alpha(&S[0][k], 32, fpx, fpy, X, Y, t0, t1);
      float al0 = fminf(amax, ex2_approx(t0)), al1 = fminf(amax, ex2_approx(t1));
      const bool c0 = live0 && al0 >= amin, c1 = live1 && al1 >= amin;
      al0 = c0 ? al0 : 0.f;
      al1 = c1 ? al1 : 0.f;
      T0 = __fsub_rn(T0, __fmul_rn(al0, T0));  // exactly as the forward rasteriser
      T1 = __fsub_rn(T1, __fmul_rn(al1, T1));
      const int j = s_pos[warp][k];
      last0 = c0 ? j : last0;
      last1 = c1 ? j : last1;
      live0 = live0 && !(T0 < tmin);
      live1 = live1 && !(T1 < tmin);
    }
  }
  int jmax = max(last0, last1);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) jmax = max(jmax, __shfl_xor_sync(0xffffffffu, jmax, o));
  if (jmax < 0) return;  // uniform over the warp; no block-wide barrier follows

  // 2. back to front
  const size_t plane = (size_t)a.H * a.W;
  const size_t po = (size_t)py * a.W + px;
  f32x2 mbar[Q], B[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    mbar[q] = pk(in0 ? a.mbar[q * plane + po] : 0.f, in1 ? a.mbar[q * plane + po + (size_t)4 * a.W] : 0.f);
    B[q] = pk(0.f, 0.f);
  }
  const bool holds = warp_sums_valid<6 + Q, 16>(lane, 6 + Q);
  const int first = (int)rg.x + (jmax - (int)rg.x) / 32 * 32;
  for (int s = first; s >= (int)rg.x; s -= 32) {
    const int n = stage((unsigned)s, true);
    for (int k = n - 1; k >= 0; --k) {
      const int j = s_pos[warp][k];
      if (j > jmax) continue;  // after the block's last composited splat
      f32x2 X, Y;
      float t0, t1;
      staged_log2_alpha(&S[0][k], 32, fpx, fpy, X, Y, t0, t1);
      const float raw0 = ex2_approx(t0), raw1 = ex2_approx(t1);  // opacity 2^-p2
      float al0 = fminf(amax, raw0), al1 = fminf(amax, raw1);
      const bool c0 = j <= last0 && al0 >= amin, c1 = j <= last1 && al1 >= amin;
      if (!__any_sync(0xffffffffu, c0 || c1)) continue;
      al0 = c0 ? al0 : 0.f;  // a pixel it does not reach: alpha 0 changes nothing below
      al1 = c1 ? al1 : 0.f;
      const float om0 = 1.f - al0, om1 = 1.f - al1;
      const f32x2 al = pk(al0, al1), om = pk(om0, om1);
      const f32x2 Tb = div2(pk(T0, T1), om);  // the transmittance before the splat
      unpk(Tb, T0, T1);
      const f32x2 w = mul2(al, Tb);
      f32x2 dal = pk(0.f, 0.f);
      float v[6 + Q];
#pragma unroll
      for (int u = 0; u < QP; ++u) {
        const ulonglong2 gg = *reinterpret_cast<const ulonglong2 *>(&S[5 + u][k]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int q = 2 * u + e;
          if (q >= Q) break;
          const f32x2 c = e ? gg.y : gg.x;
          float d0, d1;
          unpk(mul2(mbar[q], w), d0, d1);
          v[6 + q] = d0 + d1;
          dal = fma2(mbar[q], fma2(B[q], minus1, c), dal);
          B[q] = fma2(c, al, mul2(om, B[q]));
        }
      }
      float da0, da1;
      unpk(mul2(dal, Tb), da0, da1);
      // not clamped: the opacity and the exponent move alpha
      const float e0 = c0 && raw0 < amax ? da0 * raw0 : 0.f, e1 = c1 && raw1 < amax ? da1 * raw1 : 0.f;
      v[5] = (e0 + e1) * s_iopa[warp][k];  // d alpha / d opacity = 2^-p2
      const f32x2 gp = mul2(pk(e0, e1), pk(-0.6931471805599453f, -0.6931471805599453f));  // d loss / d p2
      const ulonglong2 l = *reinterpret_cast<const ulonglong2 *>(&S[4][k]);
      const ulonglong2 ab = *reinterpret_cast<const ulonglong2 *>(&S[1][k]);
      const f32x2 C = reinterpret_cast<const ulonglong2 *>(&S[2][k])->y;
      const f32x2 dx = add2(X, l.x), dy = add2(Y, l.y);
      // w = (2 A dx + B' dy, B' dx + 2 C dy): the gradient of p2, and 2 k2 times conic d
      const f32x2 wx = fma2(ab.x, add2(dx, dx), mul2(ab.y, dy)), wy = fma2(C, add2(dy, dy), mul2(ab.y, dx));
      const f32x2 gx = mul2(gp, wx), gy = mul2(gp, wy);
      float p0, p1;
#define GDGS_SUM2(I, E)  \
  unpk(E, p0, p1);       \
  v[I] = p0 + p1;
      GDGS_SUM2(0, gx)
      GDGS_SUM2(1, gy)
      GDGS_SUM2(2, mul2(gx, wx))
      GDGS_SUM2(3, mul2(gx, wy))
      GDGS_SUM2(4, mul2(gy, wy))
#undef GDGS_SUM2
      v[0] = -v[0];  // d centre = -w d p2
      v[1] = -v[1];
      int idx;
      const float sum = warp_sums<6 + Q, 16>(v, lane, 0, &idx);
      const uint32_t g = s_id[warp][k];
      if (holds) {
        if (idx < 6) atomicAdd(&a.dsplat[(size_t)g * 6 + idx], widen(sum));
        else atomicAdd(&a.dattr[(size_t)g * Q + idx - 6], sum);
      }
    }
  }
}

__global__ void __launch_bounds__(256) project_backward_kernel(ProjBwdArgs a) {
  griddep_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  const double *ds = a.dsplat + (size_t)i * 6;
  float dmx = (float)ds[0], dmy = (float)ds[1], dA = (float)ds[2], dB = (float)ds[3], dC = (float)ds[4],
        dopa = (float)ds[5];
  float gm[3] = {0.f, 0.f, 0.f}, gs[3] = {0.f, 0.f, 0.f}, gq[4] = {0.f, 0.f, 0.f, 0.f};
  const bool any = dmx != 0.f || dmy != 0.f || dA != 0.f || dB != 0.f || dC != 0.f || dopa != 0.f;
  if (any) {
    const float *w = a.w2c;
    const float mx = a.mean[3 * i], my = a.mean[3 * i + 1], mz = a.mean[3 * i + 2];
    const float s0 = a.scale[3 * i], s1 = a.scale[3 * i + 1], s2 = a.scale[3 * i + 2];
    float qr[4] = {a.quat[4 * i], a.quat[4 * i + 1], a.quat[4 * i + 2], a.quat[4 * i + 3]};
    const float qlen = sqrtf(qr[0] * qr[0] + qr[1] * qr[1] + qr[2] * qr[2] + qr[3] * qr[3]);
    const float qw = qr[0] / qlen, qx = qr[1] / qlen, qy = qr[2] / qlen, qz = qr[3] / qlen;
    float R[3][3] = {{1.f - 2.f * (qy * qy + qz * qz), 2.f * (qx * qy - qw * qz), 2.f * (qx * qz + qw * qy)},
                     {2.f * (qx * qy + qw * qz), 1.f - 2.f * (qx * qx + qz * qz), 2.f * (qy * qz - qw * qx)},
                     {2.f * (qx * qz - qw * qy), 2.f * (qy * qz + qw * qx), 1.f - 2.f * (qx * qx + qy * qy)}};
    const float sv[3] = {s0, s1, s2};
    float M[3][3], Sig[3][3];
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) M[r][c] = R[r][c] * sv[c];
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) Sig[r][c] = M[r][0] * M[c][0] + M[r][1] * M[c][1] + M[r][2] * M[c][2];
    const float tx = w[0] * mx + w[1] * my + w[2] * mz + w[3];
    const float ty = w[4] * mx + w[5] * my + w[6] * mz + w[7];
    const float tz = w[8] * mx + w[9] * my + w[10] * mz + w[11];
    const float iz = 1.f / tz;
    float J[2][3] = {{a.fx * iz, 0.f, -a.fx * tx * iz * iz}, {0.f, a.fy * iz, -a.fy * ty * iz * iz}};
    float Tm[2][3];
    for (int r = 0; r < 2; ++r)
      for (int c = 0; c < 3; ++c) Tm[r][c] = J[r][0] * w[c] + J[r][1] * w[4 + c] + J[r][2] * w[8 + c];
    float TS[2][3];
    for (int r = 0; r < 2; ++r)
      for (int c = 0; c < 3; ++c) TS[r][c] = Tm[r][0] * Sig[0][c] + Tm[r][1] * Sig[1][c] + Tm[r][2] * Sig[2][c];
    // d Sigma2D = -C (sum g k2 d d^T) C with the moments of w = 2 k2 C d
    const float k2 = a.exp_coef * 1.4426950408889634f;
    const float ms = -1.f / (4.f * k2);
    const float Sb[2][2] = {{ms * dA, ms * dB}, {ms * dB, ms * dC}};
    // d T = 2 Sb T Sigma
    float Tb[2][3];
    for (int r = 0; r < 2; ++r)
      for (int c = 0; c < 3; ++c) Tb[r][c] = 2.f * (Sb[r][0] * TS[0][c] + Sb[r][1] * TS[1][c]);
    // d J = d T W_R^T
    float Jb[2][3];
    for (int r = 0; r < 2; ++r)
      for (int c = 0; c < 3; ++c) Jb[r][c] = Tb[r][0] * w[4 * c] + Tb[r][1] * w[4 * c + 1] + Tb[r][2] * w[4 * c + 2];
    float tb[3];
    tb[0] = dmx * a.fx * iz + Jb[0][2] * (-a.fx * iz * iz);
    tb[1] = dmy * a.fy * iz + Jb[1][2] * (-a.fy * iz * iz);
    tb[2] = dmx * (-a.fx * tx * iz * iz) + dmy * (-a.fy * ty * iz * iz) +
            Jb[0][0] * (-a.fx * iz * iz) + Jb[0][2] * (2.f * a.fx * tx * iz * iz * iz) +
            Jb[1][1] * (-a.fy * iz * iz) + Jb[1][2] * (2.f * a.fy * ty * iz * iz * iz);
    for (int c = 0; c < 3; ++c) gm[c] = w[c] * tb[0] + w[4 + c] * tb[1] + w[8 + c] * tb[2];
    // Sigma = R diag(s^2) R^T. In the splat's own frame d Sigma is G = B^T Sb B, B = T R:
    // d s_k = 2 s_k G_kk, and turning the frame by w (R exp[w]) changes the loss by t . w
    // with t_1 = 2 G_23 (s_2^2 - s_3^2) and cyclic. The quaternion's gradient is
    // 2 q (0, t) / |q|. (Through d R it would be a difference of terms s_i^2 G_ij that
    // nearly cancel for nearly round splats, and of its own component along q.)
    float Bm[2][3], G[3][3];
    for (int r = 0; r < 2; ++r)
      for (int c = 0; c < 3; ++c) Bm[r][c] = Tm[r][0] * R[0][c] + Tm[r][1] * R[1][c] + Tm[r][2] * R[2][c];
    for (int r = 0; r < 3; ++r)
      for (int c = r; c < 3; ++c)
        G[r][c] = Bm[0][r] * (Sb[0][0] * Bm[0][c] + Sb[0][1] * Bm[1][c]) +
                  Bm[1][r] * (Sb[1][0] * Bm[0][c] + Sb[1][1] * Bm[1][c]);
    for (int c = 0; c < 3; ++c) gs[c] = 2.f * sv[c] * G[c][c];
    const float t0 = 2.f * G[1][2] * ((s1 - s2) * (s1 + s2)), t1 = 2.f * G[0][2] * ((s2 - s0) * (s2 + s0)),
                t2 = 2.f * G[0][1] * ((s0 - s1) * (s0 + s1));
    const float q2 = 2.f / qlen;
    gq[0] = -q2 * (qx * t0 + qy * t1 + qz * t2);
    gq[1] = q2 * (qw * t0 + qy * t2 - qz * t1);
    gq[2] = q2 * (qw * t1 + qz * t0 - qx * t2);
    gq[3] = q2 * (qw * t2 + qx * t1 - qy * t0);
  }
  for (int c = 0; c < 3; ++c) a.d_mean[3 * i + c] = gm[c];
  for (int c = 0; c < 3; ++c) a.d_scale[3 * i + c] = gs[c];
  for (int c = 0; c < 4; ++c) a.d_quat[4 * i + c] = gq[c];
  a.d_opacity[i] = dopa;
}

}  // namespace

cudaError_t launch_divergence_adjoint(const DivAdjArgs &a, cudaStream_t st) {
  const size_t total = (size_t)a.C * a.H * a.W;
  int blocks = (int)((total + 255) / 256);
  if (blocks > 8192) blocks = 8192;
  { LaunchScope ls_("divergence_adjoint", st); launch_k(divergence_adjoint_kernel, blocks, 256, 0, st, a); }
  return cudaGetLastError();
}

cudaError_t launch_raster_backward(const RasterBwdArgs &a, cudaStream_t st) {
  if (a.T == 0) return cudaSuccess;
  LaunchScope ls_("raster_backward", st);
  switch (a.Q) {
    case 1: launch_k(raster_backward_kernel<1>, a.T, kBwdThreads, 0, st, a); break;
    case 2: launch_k(raster_backward_kernel<2>, a.T, kBwdThreads, 0, st, a); break;
    case 3: launch_k(raster_backward_kernel<3>, a.T, kBwdThreads, 0, st, a); break;
    case 4: launch_k(raster_backward_kernel<4>, a.T, kBwdThreads, 0, st, a); break;
    case 6: launch_k(raster_backward_kernel<6>, a.T, kBwdThreads, 0, st, a); break;
    case 8: launch_k(raster_backward_kernel<8>, a.T, kBwdThreads, 0, st, a); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_project_backward(const ProjBwdArgs &a, cudaStream_t st) {
  if (a.n == 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((a.n + 255) / 256);
  { LaunchScope ls_("project_backward", st); launch_k(project_backward_kernel, blocks, 256, 0, st, a); }
  return cudaGetLastError();
}

}  // namespace gdgs
