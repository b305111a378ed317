// The passes of the direct solve, one set of kernels per FFT length (fct.cu describes
// the solve). A length is a product of two to four radices that are template arguments,
// so all strides, twiddle steps and thread counts are constants and every shared-memory
// access is one base register plus an immediate; a kernel that picked the radix at run
// time kept every radix's registers live and spilled 1.4 KB per thread.
//
// The lengths (end of this file) are the even products of two or three radices up to
// 16, each with the fewest stages and then the fewest threads; a subset, and a few of
// four radices, serve Bluestein's convolution for the other sides.
#pragma once

#include "fct.cuh"

namespace gdgs {

namespace {

// ------------------------------------------------------------------ small DFTs

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// Cosines and sines of 2 pi j / R of the radices that need them, in constant memory:
// the multiply-adds take them as constant-bank operands, while literals would be kept in
// registers across the stage loop.
struct Trig {
  float c3[3], s3[3];
  float c5[5], s5[5];
  float c8[8], s8[8];
  float c9[9], s9[9];
  float c16[16], s16[16];
};
__constant__ Trig kTrig = {
    {1.0f, -0.5f, -0.5f},
    {0.0f, 0.866025404f, -0.866025404f},
    {1.0f, 0.309016994f, -0.809016994f, -0.809016994f, 0.309016994f},
    {0.0f, 0.951056516f, 0.587785252f, -0.587785252f, -0.951056516f},
    {1.0f, 0.707106781f, 0.0f, -0.707106781f, -1.0f, -0.707106781f, 0.0f, 0.707106781f},
    {0.0f, 0.707106781f, 1.0f, 0.707106781f, 0.0f, -0.707106781f, -1.0f, -0.707106781f},
    {1.0f, 0.766044443f, 0.173648178f, -0.5f, -0.939692621f, -0.939692621f, -0.5f, 0.173648178f, 0.766044443f},
    {0.0f, 0.64278761f, 0.984807753f, 0.866025404f, 0.342020143f, -0.342020143f, -0.866025404f, -0.984807753f, -0.64278761f},
    {1.0f, 0.923879533f, 0.707106781f, 0.382683432f, 0.0f, -0.382683432f, -0.707106781f, -0.923879533f, -1.0f, -0.923879533f, -0.707106781f, -0.382683432f, 0.0f, 0.382683432f, 0.707106781f, 0.923879533f},
    {0.0f, 0.382683432f, 0.707106781f, 0.923879533f, 1.0f, 0.923879533f, 0.707106781f, 0.382683432f, 0.0f, -0.382683432f, -0.707106781f, -0.923879533f, -1.0f, -0.923879533f, -0.707106781f, -0.382683432f},
};

template <int P>
__device__ __forceinline__ float trig_c(int i) {
  if constexpr (P == 3) return kTrig.c3[i];
  if constexpr (P == 5) return kTrig.c5[i];
  if constexpr (P == 8) return kTrig.c8[i];
  if constexpr (P == 9) return kTrig.c9[i];
  if constexpr (P == 16) return kTrig.c16[i];
}
template <int P>
__device__ __forceinline__ float trig_s(int i) {
  if constexpr (P == 3) return kTrig.s3[i];
  if constexpr (P == 5) return kTrig.s5[i];
  if constexpr (P == 8) return kTrig.s8[i];
  if constexpr (P == 9) return kTrig.s9[i];
  if constexpr (P == 16) return kTrig.s16[i];
}

template <int R>
struct Dft;

template <>
struct Dft<2> {
  static __device__ __forceinline__ void run(float2 (&v)[2]) {
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <>
struct Dft<4> {
  static __device__ __forceinline__ void run(float2 (&v)[4]) {
    const float2 a = cadd(v[0], v[2]), b = csub(v[0], v[2]), c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
    v[0] = cadd(a, c);
    v[2] = csub(a, c);
    v[1] = make_float2(b.x + d.y, b.y - d.x);
    v[3] = make_float2(b.x - d.y, b.y + d.x);
  }
};

// Odd primes: X_m = A_m - i B_m, X_{P-m} = A_m + i B_m with A_m = x_0 + sum cos (x_j +
// x_{P-j}), B_m = sum sin (x_j - x_{P-j}).
template <int P>
struct DftPrime {
  static __device__ __forceinline__ void run(float2 (&v)[P]) {
    constexpr int h = (P - 1) / 2;
    float2 sm[h], df[h];
    float2 x0 = v[0];
#pragma unroll
    for (int j = 1; j <= h; ++j) {
      sm[j - 1] = cadd(v[j], v[P - j]);
      df[j - 1] = csub(v[j], v[P - j]);
    }
    float2 t = x0;
#pragma unroll
    for (int j = 0; j < h; ++j) t = cadd(t, sm[j]);
    v[0] = t;
#pragma unroll
    for (int m = 1; m <= h; ++m) {
      float2 a = x0, b = make_float2(0.f, 0.f);
#pragma unroll
      for (int j = 1; j <= h; ++j) {
        const int i = (j * m) % P;
        a.x = fmaf(trig_c<P>(i), sm[j - 1].x, a.x);
        a.y = fmaf(trig_c<P>(i), sm[j - 1].y, a.y);
        b.x = fmaf(trig_s<P>(i), df[j - 1].x, b.x);
        b.y = fmaf(trig_s<P>(i), df[j - 1].y, b.y);
      }
      v[m] = make_float2(a.x + b.y, a.y - b.x);
      v[P - m] = make_float2(a.x - b.y, a.y + b.x);
    }
  }
};
template <> struct Dft<3> : DftPrime<3> {};
template <> struct Dft<5> : DftPrime<5> {};

// Coprime factors (Good-Thomas): index maps only, no twiddles.
constexpr int inv_mod(int a, int m) {
  for (int i = 1; i < m; ++i)
    if ((a * i) % m == 1) return i;
  return 1;
}
template <int R1, int R2>
struct DftPfa {
  static constexpr int R = R1 * R2;
  static constexpr int U1 = R2 * inv_mod(R2 % R1, R1), U2 = R1 * inv_mod(R1 % R2, R2);
  static __device__ __forceinline__ void run(float2 (&v)[R]) {
    float2 w[R];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) {
      float2 t[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) t[n1] = v[(R2 * n1 + R1 * n2) % R];
      Dft<R1>::run(t);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) w[k1 * R2 + n2] = t[k1];
    }
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      float2 t[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) t[n2] = w[k1 * R2 + n2];
      Dft<R2>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2)
        v[(k1 * U1 + k2 * U2) % R] = t[k2];
    }
  }
};
template <> struct Dft<6> : DftPfa<2, 3> {};
template <> struct Dft<10> : DftPfa<2, 5> {};
template <> struct Dft<12> : DftPfa<4, 3> {};
template <> struct Dft<15> : DftPfa<3, 5> {};

// Equal prime factors (Cooley-Tukey): n = R2 n1 + n2, k = k1 + R1 k2, twiddles W_R^{n2 k1}.
template <int R>
__device__ __forceinline__ float2 ct_twiddle(int e) {
  return make_float2(trig_c<R>(e), -trig_s<R>(e));
}
template <int R1, int R2>
struct DftCt {
  static constexpr int R = R1 * R2;
  static __device__ __forceinline__ void run(float2 (&v)[R]) {
    float2 w[R];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) {
      float2 t[R1];
#pragma unroll
      for (int n1 = 0; n1 < R1; ++n1) t[n1] = v[R2 * n1 + n2];
      Dft<R1>::run(t);
#pragma unroll
      for (int k1 = 0; k1 < R1; ++k1) w[k1 * R2 + n2] = n2 * k1 == 0 ? t[k1] : cmul(t[k1], ct_twiddle<R>((n2 * k1) % R));
    }
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      float2 t[R2];
#pragma unroll
      for (int n2 = 0; n2 < R2; ++n2) t[n2] = w[k1 * R2 + n2];
      Dft<R2>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < R2; ++k2) v[k1 + R1 * k2] = t[k2];
    }
  }
};
template <> struct Dft<8> : DftCt<2, 4> {};
template <> struct Dft<9> : DftCt<3, 3> {};
template <> struct Dft<16> : DftCt<4, 4> {};

// ------------------------------------------------------------------ FFT in shared memory

constexpr int ceil_div(int a, int b) { return (a + b - 1) / b; }
constexpr int cmax(int a, int b) { return a > b ? a : b; }
constexpr int cmin(int a, int b) { return a < b ? a : b; }
constexpr int stage_threads(int len, int r) { return r > 1 ? ceil_div(len / r, 16 / r) : 1; }

// Extra shared-memory wavefronts of a half-warp's 8-byte stores when element i of a
// stage's output (blocks of `blk` elements, `p` slots of padding after each) goes to slot
// (i + i / blk * p) * mult (+ the transform, for mult interleaved ones): the stage's
// threads j write i = j / ns * blk + j % ns.
constexpr int store_conflicts(int ns, int blk, int p, int mult) {
  int worst = 0;
  for (int j0 = 0; j0 < 64; j0 += 16 / cmin(mult, 16)) {
    int bank[16] = {};
    for (int l = 0; l < 16; ++l) {
      const int j = j0 + l / cmin(mult, 16), g = l % cmin(mult, 16);
      ++bank[((j / ns * (blk + p) + j % ns) * mult + g) % 16];
    }
    int m = 0;
    for (int b = 0; b < 16; ++b) m = cmax(m, bank[b]);
    worst += m - 1;
  }
  return worst;
}
constexpr int best_pad(int ns, int blk, int mult) {
  int best = 0, conflicts = 1 << 30;
  for (int p = 0; p < 16; ++p)
    if (store_conflicts(ns, blk, p, mult) < conflicts) {
      conflicts = store_conflicts(ns, blk, p, mult);
      best = p;
    }
  return best;
}

template <int N>
struct Num {
  static constexpr int value = N;
};

// The inputs j, j + M, ... of a first-stage butterfly from f(i).
template <int M, int R, class Fn>
__device__ __forceinline__ void gather(float2 (&v)[R], int j, const Fn &f) {
#pragma unroll
  for (int r = 0; r < R; ++r) v[r] = f(j + r * M);
}

// One Stockham stage, in place: thread t of the TP threads of a transform reads its
// butterflies (up to 16 points) into registers, all threads meet, and it writes them to
// their places. Input i is at slot i + i / IB * IP, output i at i + i / (NS R) * OP. The
// first stage gathers through load(v, j, M), the last may write through store(i, v). The
// twiddles of inputs 4a + b are products of two table values, which keeps their error at
// a few roundings.
struct NoStore {
  static constexpr bool global = false;
};
template <int R, int NS, int LEN, int TP, int IB, int IP, int OP, int MULT, class Load, class Store>
__device__ __forceinline__ void fft_stage(float2 *S, const float2 *__restrict__ tw, int t, bool meet,
                                          const Load &load, const Store &store) {
  constexpr int M = LEN / R, MB = (M + TP - 1) / TP, STEP = LEN / (NS * R);
  static_assert(MB * R <= 16, "points per thread");
  float2 v[MB][R];
#pragma unroll
  for (int b = 0; b < MB; ++b) {
    const int j = t + b * TP;
    if (t < TP && (MB * TP == M || j < M)) {
      if constexpr (NS == 1) {
        load(v[b], j, Num<M>{});
      } else {
        static_assert(M % IB == 0, "whole blocks between the inputs of a butterfly");
        const float2 *s = S + (j + (IP ? j / IB * IP : 0)) * MULT;
#pragma unroll
        for (int r = 0; r < R; ++r) v[b][r] = s[r * (M + M / IB * IP) * MULT];
      }
    }
  }
  if (meet) __syncthreads();
#pragma unroll
  for (int b = 0; b < MB; ++b) {
    const int j = t + b * TP;
    if (t < TP && (MB * TP == M || j < M)) {
      const int q = j / NS, k = j - q * NS;
      if constexpr (NS > 1) {
        const float2 *wk = tw + k * STEP;
        float2 w[4];
        w[1] = __ldg(wk);
        w[2] = cmul(w[1], w[1]);
        w[3] = cmul(w[2], w[1]);
#pragma unroll
        for (int r = 1; r < R; ++r) {
          if (r < 4) {
            v[b][r] = cmul(v[b][r], w[r]);
          } else if ((r & 3) == 0) {
            const float2 wa = __ldg(tw + r * k * STEP);
            v[b][r] = cmul(v[b][r], wa);
#pragma unroll
            for (int e = 1; e < 4; ++e)
              if (r + e < R) v[b][r + e] = cmul(v[b][r + e], cmul(wa, w[e]));
          }
        }
      }
      Dft<R>::run(v[b]);
      if constexpr (Store::global) {
#pragma unroll
        for (int r = 0; r < R; ++r) store(q * NS * R + k + r * NS, v[b][r]);
      } else {
        float2 *s = S + (q * (NS * R + OP) + k) * MULT;
#pragma unroll
        for (int r = 0; r < R; ++r) s[r * NS * MULT] = v[b][r];
      }
    }
  }
  if constexpr (!Store::global) __syncthreads();
}

// MULT transforms interleaved (element slot e of transform g at e * MULT + g).
template <int R1, int R2, int R3, int R4>
struct Fft {
  static constexpr int LEN = R1 * R2 * R3 * R4;
  static constexpr int STAGES = 2 + (R3 > 1) + (R4 > 1);
  static constexpr int TP = cmax(cmax(stage_threads(LEN, R1), stage_threads(LEN, R2)),
                                 cmax(stage_threads(LEN, R3), stage_threads(LEN, R4)));
  // transforms per block: rows about 256 threads (128 and 512 were 1-6 % slower); columns
  // the power of two of pairs that gives at most 384 threads (256 or 768: 5-40 % slower)
  static constexpr int G_ROWS = cmax(1, 256 / TP);
  static constexpr int cols_g() {
    int g = 1;
    while (g < 32 && 2 * g * TP <= 384) g *= 2;
    return g;
  }
  static constexpr int G_COLS = cols_g();
  template <int MULT>
  struct Layout {
    static constexpr int P1 = best_pad(1, R1, MULT);
    static constexpr int P2 = R3 > 1 ? best_pad(R1, R1 * R2, MULT) : 0;
    static constexpr int P3 = R4 > 1 ? best_pad(R1 * R2, R1 * R2 * R3, MULT) : 0;
    static constexpr int SLOTS =
        (cmax(cmax(LEN + LEN / R1 * P1, LEN + LEN / (R1 * R2) * P2), LEN + LEN / (R1 * R2 * R3) * P3) + 1) / 2 * 2;
  };
  // The forward DFT of what load() gathers: the first write into S waits for all threads when
  // `meet` (S is still being read); the result goes to S in natural order or to store().
  template <int MULT, class Load, class Store>
  static __device__ __forceinline__ void run(float2 *S, const float2 *tw, int t, bool meet, const Load &load,
                                             const Store &store) {
    using L = Layout<MULT>;
    NoStore none;
    fft_stage<R1, 1, LEN, TP, 1, 0, L::P1, MULT>(S, tw, t, meet, load, none);
    if constexpr (R3 == 1) {
      fft_stage<R2, R1, LEN, TP, R1, L::P1, 0, MULT>(S, tw, t, true, load, store);
    } else {
      fft_stage<R2, R1, LEN, TP, R1, L::P1, L::P2, MULT>(S, tw, t, true, load, none);
      if constexpr (R4 == 1) {
        fft_stage<R3, R1 * R2, LEN, TP, R1 * R2, L::P2, 0, MULT>(S, tw, t, true, load, store);
      } else {
        fft_stage<R3, R1 * R2, LEN, TP, R1 * R2, L::P2, L::P3, MULT>(S, tw, t, true, load, none);
        fft_stage<R4, R1 * R2 * R3, LEN, TP, R1 * R2 * R3, L::P3, 0, MULT>(S, tw, t, true, load, store);
      }
    }
  }
};

template <class F>
struct StoreTo {
  static constexpr bool global = true;
  F f;
  __device__ __forceinline__ void operator()(int i, float2 v) const { f(i, v); }
};
template <class F>
__device__ __forceinline__ StoreTo<F> store_to(const F &f) {
  return StoreTo<F>{f};
}

// Cosine coefficients k and n - k of the two real sequences packed in Z (z = Z[k], zn =
// Z[n-k]; (c, s) of pi k / 2n), DCT-II without scaling.
struct Quad {
  float ak, an, bk, bn;
};
__device__ __forceinline__ Quad dct_post(float2 z, float2 zn, float2 th) {
  const float sp = 0.5f * (z.x + zn.x), sm = 0.5f * (z.x - zn.x);
  const float tp = 0.5f * (z.y + zn.y), tm = 0.5f * (z.y - zn.y);
  Quad q;
  q.ak = fmaf(th.x, sp, th.y * tm);
  q.an = fmaf(th.y, sp, -th.x * tm);
  q.bk = fmaf(th.x, tp, -th.y * sm);
  q.bn = fmaf(th.y, tp, th.x * sm);
  return q;
}
// The inverse: packed values whose forward DFT (parts swapped) gives the two sequences.
__device__ __forceinline__ void dct_pre(const Quad &q, float2 th, float2 &z, float2 &zn) {
  const float ar = fmaf(th.x, q.ak, th.y * q.an), ai = fmaf(th.y, q.ak, -th.x * q.an);
  const float br = fmaf(th.x, q.bk, th.y * q.bn), bi = fmaf(th.y, q.bk, -th.x * q.bn);
  z = make_float2(ai + br, ar - bi);   // swapped (im, re) of Va + i Vb
  zn = make_float2(br - ai, ar + bi);  // and of conj(Va) + i conj(Vb)
}

// ------------------------------------------------------------------ the passes

// Values j and j + 1 of a row (j even; the second is `pad` where the row ends at j).
__device__ __forceinline__ float2 ld_pair(const float *row, int j, int W) {
  if ((W & 1) == 0) return __ldg(reinterpret_cast<const float2 *>(row + j));
  const float a = __ldg(row + j);
  return make_float2(a, j + 1 < W ? __ldg(row + j + 1) : a);
}
__device__ __forceinline__ void st_pair(float *row, int j, int W, float2 v) {
  if ((W & 1) == 0) {
    *reinterpret_cast<float2 *>(row + j) = v;
  } else {
    row[j] = v.x;
    if (j + 1 < W) row[j + 1] = v.y;
  }
}

// A row pair's columns j, j + 1 with every neighbour the residual needs (a neighbour
// outside the image is the pixel itself).
struct Patch {
  float2 a, b, n, s;      // rows ia, ib, and the ones above and below
  float al, ar, bl, br;   // columns j - 1 and j + 2 of rows ia, ib
};
__device__ __forceinline__ Patch ld_patch(const float *u, int ia, int j, int W, int H) {
  Patch p;
  const float *ra = u + (size_t)ia * W, *rb = ra + W;
  const bool vb = ia + 1 < H;
  p.a = ld_pair(ra, j, W);
  p.b = vb ? ld_pair(rb, j, W) : p.a;
  p.n = ia > 0 ? ld_pair(ra - W, j, W) : p.a;
  p.s = ia + 2 < H ? ld_pair(rb + W, j, W) : p.b;
  p.al = j > 0 ? __ldg(ra + j - 1) : p.a.x;
  p.ar = j + 2 < W ? __ldg(ra + j + 2) : p.a.y;
  p.bl = !vb ? 0.f : j > 0 ? __ldg(rb + j - 1) : p.b.x;
  p.br = !vb ? 0.f : j + 2 < W ? __ldg(rb + j + 2) : p.b.y;
  return p;
}

// Bluestein's chirp factors on a value going into the DFT and coming out of it (where the
// parts are swapped: the second FFT is an inverse one).
__device__ __forceinline__ float2 chirp_out(float2 z, float2 w, float inv_len) {
  const float2 v = cmul(make_float2(z.y, z.x), w);
  return make_float2(v.x * inv_len, v.y * inv_len);
}

// The DFT of the n points that src() gathers into S (natural order; a Bluestein result through
// chirp_out). SMEM: src reads S.
template <class F, bool BL, int MULT, class Src>
__device__ __forceinline__ void dft(float2 *S, const FctSide &d, int t, bool smem, const Src &src) {
  if constexpr (!BL) {
    F::template run<MULT>(S, d.tw, t, smem, src, NoStore{});
  } else {
    F::template run<MULT>(S, d.tw, t, smem, [&](auto &v, int j, auto step) {
      constexpr int M = decltype(step)::value;
      src(v, j, step);
#pragma unroll
      for (int r = 0; r < (int)(sizeof(v) / sizeof(v[0])); ++r) {
        const int i = j + r * M;
        if (i < d.n) v[r] = cmul(v[r], __ldg(d.chirp + i));
        else v[r] = make_float2(0.f, 0.f);
      }
    }, NoStore{});
    // opaque, or what both FFTs have in common (twiddles, addresses) stays in registers
    // from one to the other
    asm volatile("" : "+r"(t));
    F::template run<MULT>(S, d.tw, t, true, [&](auto &v, int j, auto step) {
      gather<decltype(step)::value>(v, j, [&](int i) -> float2 {
        const float2 w = cmul(S[i * MULT], __ldg(d.bhat + i));
        return make_float2(w.y, w.x);  // an inverse FFT is a forward one with the parts swapped
      });
    }, NoStore{});
  }
}

// Blocks per SM the register budget is set for: the passes wait for loads, barriers and
// twiddles more than they issue, so more warps pay. Measured at 3840x2160x3, rows + columns + rows
// back of a solve: 56 registers 652 us, 64 670 us, 80 704 us, 48 655 us (and slower at 1080p).
constexpr int blocks_per_sm(int threads) { return cmax(1, 65536 / (56 * ceil_div(threads, 32) * 32)); }

// Rows forward (kc: cycle; cycle 0 transforms rho less the high part of its mean, later ones the
// residual of the iterate; cycles 0 and 1 record the norm of what they transform).
template <class F, bool BL>
__global__ void __launch_bounds__(ceil_div(F::G_ROWS * F::TP, 32) * 32, blocks_per_sm(F::G_ROWS * F::TP))
fct_rows_kernel(const __grid_constant__ FctArgs a, int kc) {
  griddep_enter();
  extern __shared__ float2 fct_sm[];
  constexpr int TP = F::TP, G = F::G_ROWS;
  const int c = blockIdx.y;
  // the residual after one cycle is recorded by this launch itself (kc == 1), after two by
  // the finalize pass before it
  const FctChannel ch = fct_block_channel(a, c, kc == 0 ? kFctRows : kc == 1 ? 0 : kc);
  if (ch.skip) return;
  const int g = threadIdx.x / TP, t = g < G ? (int)threadIdx.x - g * TP : TP;
  float2 *S = fct_sm + (g < G ? g : 0) * F::template Layout<1>::SLOTS;
  const int W = a.W, H = a.H;
  const size_t plane = (size_t)H * W;
  const int ia = 2 * (blockIdx.x * G + g);
  const bool va = t < TP && ia < H, vb = t < TP && ia + 1 < H;
  const float *rho = a.rho + c * plane;
  float acc = 0.f;
  if (kc > 0) {
    const float *uh = a.uhi + c * plane, *ul = a.ulo + c * plane;
    // L u of the part u at columns j, j + 1 of both rows
    auto lap = [&](const float *u, int j, float2 &la, float2 &lb) {
      const Patch h = ld_patch(u, ia, j, W, H);
      la = make_float2(fct_lap(h.a.x, h.a.y, h.al, h.b.x, h.n.x), fct_lap(h.a.y, h.ar, h.a.x, h.b.y, h.n.y));
      lb = make_float2(fct_lap(h.b.x, h.b.y, h.bl, h.s.x, h.a.x), fct_lap(h.b.y, h.br, h.b.x, h.s.y, h.a.y));
    };
    if (t < TP) {
#pragma unroll 2
      for (int m = t; m < (W + 1) / 2; m += TP) {
        const int j = 2 * m;
        float2 ra = make_float2(0.f, 0.f), rb = ra;
        if (va) {
          float2 la, lb;
          ra = ld_pair(rho + (size_t)ia * W, j, W);
          if (vb) rb = ld_pair(rho + (size_t)(ia + 1) * W, j, W);
          FctResidual r[4] = {{ra.x, ch.hi, ch.lo}, {ra.y, ch.hi, ch.lo}, {rb.x, ch.hi, ch.lo}, {rb.y, ch.hi, ch.lo}};
          auto minus_lap = [&](const float *u) {
            lap(u, j, la, lb);
            r[0].minus(la.x);
            r[1].minus(la.y);
            r[2].minus(lb.x);
            r[3].minus(lb.y);
          };
          minus_lap(uh);
          if (kc > 1) minus_lap(ul);
          ra = make_float2(r[0].value(), r[1].value());
          rb = make_float2(r[2].value(), r[3].value());
          if (!vb) rb = make_float2(0.f, 0.f);
          acc = fmaf(ra.x, ra.x, acc);
          acc = fmaf(rb.x, rb.x, acc);
          if (j + 1 < W) {
            acc = fmaf(ra.y, ra.y, acc);
            acc = fmaf(rb.y, rb.y, acc);
          }
        }
        S[m] = make_float2(ra.x, rb.x);
        if (j + 1 < W) S[W - 1 - m] = make_float2(ra.y, rb.y);
      }
    }
    __syncthreads();
  }
  // point n of the DFT: column 2n (first half) or 2 (W - 1 - n) + 1, of rows ia and ia + 1
  const float *ra = rho + (size_t)ia * W;
  dft<F, BL, 1>(S, a.x, t, kc > 0, [&](auto &v, int j0, auto step) {
    constexpr int M = decltype(step)::value;
    if (kc > 0) {
      gather<M>(v, j0, [&](int i) { return BL && i >= W ? make_float2(0.f, 0.f) : S[i]; });
    } else {
      gather<M>(v, j0, [&](int i) -> float2 {
        if (BL && i >= W) return make_float2(0.f, 0.f);
        const int j = 2 * i < W ? 2 * i : 2 * (W - 1 - i) + 1;
        const float2 r = make_float2(va ? __ldg(ra + j) - ch.hi : 0.f, vb ? __ldg(ra + W + j) - ch.hi : 0.f);
        acc = fmaf(r.x, r.x, fmaf(r.y, r.y, acc));
        return r;
      });
    }
  });
  if (va) {
    constexpr float inv_len = 1.f / (float)F::LEN;
    float *sa = a.spec + ((size_t)c * H + ia) * a.wp, *sb = sa + a.wp;
    for (int k = t; k <= W / 2; k += TP) {
      const int kn = k == 0 ? 0 : W - k;
      float2 z = S[k], zn = S[kn];
      if (BL) {
        z = chirp_out(z, __ldg(a.x.chirp + k), inv_len);
        zn = chirp_out(zn, __ldg(a.x.chirp + kn), inv_len);
      }
      const Quad q = dct_post(z, zn, __ldg(a.x.th + k));
      sa[k] = q.ak;
      if (k > 0) sa[kn] = q.an;
      if (vb) {
        sb[k] = q.bk;
        if (k > 0) sb[kn] = q.bn;
      }
    }
  }
  if (kc <= 1) {
    acc = fct_block_sum(acc);
    if (threadIdx.x == 0) atomicAdd(&a.ctrl->rnorm2[kc == 0 ? fct_sq_slot(c) : fct_slot(1, c)], (double)acc);
  }
}

// Columns: DCT along y of G column pairs, the division by lambda, and back.
template <class F, bool BL>
__global__ void __launch_bounds__(ceil_div(F::G_COLS * F::TP, 32) * 32, blocks_per_sm(F::G_COLS * F::TP))
fct_cols_kernel(const __grid_constant__ FctArgs a, int kc) {
  griddep_enter();
  extern __shared__ float2 fct_sm[];
  constexpr int TP = F::TP, G = F::G_COLS;
  const int c = blockIdx.y;
  if (fct_block_skip(a, c, kc == 0 ? kFctFirst : kc)) return;
  const int g = threadIdx.x % G;
  const int t = min((int)threadIdx.x / G, TP);
  float2 *S = fct_sm + g;
  const int W = a.W, H = a.H;
  const int ja = 2 * (G * blockIdx.x + g);
  const bool in = ja < W;
  float *col = a.spec + (size_t)c * H * a.wp + (in ? ja : 0);
  const int wp = a.wp;
  constexpr float inv_len = 1.f / (float)F::LEN;
  // point n of the DFT: row 2n (first half) or 2 (H - 1 - n) + 1
  auto row_of = [&](int i) { return 2 * i < H ? 2 * i : 2 * (H - 1 - i) + 1; };
  auto from_image = [&](int i) -> float2 {
    float2 z = make_float2(0.f, 0.f);
    if (in && (!BL || i < H)) z = __ldcg(reinterpret_cast<const float2 *>(col + (size_t)row_of(i) * wp));
    if (ja + 1 >= W) z.y = 0.f;
    return z;
  };
  auto to_image = [&](int i, float2 v) {
    if (BL) {
      if (i >= H) return;
      v = chirp_out(v, __ldg(a.y.chirp + i), inv_len);
    }
    if (in) *reinterpret_cast<float2 *>(col + (size_t)row_of(i) * wp) = make_float2(v.y, v.x);
  };
  // the spectral step on points k and H - k of both columns (and the sum of squares that sets
  // the grid of the correction)
  float acc = 0.f;
  auto spectral = [&] {
    if (t < TP) {
      const float lxa = in ? __ldg(a.x.s2 + ja) : 1.f, lxb = ja + 1 < W ? __ldg(a.x.s2 + ja + 1) : 1.f;
      const float scale = -1.f / ((float)W * (float)H);
      for (int k = t; k <= H / 2; k += TP) {
        const int kn = k == 0 ? 0 : H - k;
        const float2 tk = __ldg(a.y.th + k);
        float2 z = S[k * G], zn = S[kn * G];
        if (BL) {
          z = chirp_out(z, __ldg(a.y.chirp + k), inv_len);
          zn = chirp_out(zn, __ldg(a.y.chirp + kn), inv_len);
        }
        Quad q = dct_post(z, zn, tk);
        const float lk = __ldg(a.y.s2 + k), ln = __ldg(a.y.s2 + kn);
        if (k == 0 && ja == 0) a.ctrl->rho_mean[c] += -scale * q.ak;  // (one thread)
        q.ak = (k == 0 && ja == 0) ? 0.f : q.ak * __fdividef(scale, lk + lxa);
        q.bk = q.bk * __fdividef(scale, lk + lxb);
        q.an = k == 0 ? 0.f : q.an * __fdividef(scale, ln + lxa);
        q.bn = k == 0 ? 0.f : q.bn * __fdividef(scale, ln + lxb);
        if (in) acc = fmaf(q.ak, q.ak, fmaf(q.an, q.an, acc));
        if (ja + 1 < W) acc = fmaf(q.bk, q.bk, fmaf(q.bn, q.bn, acc));
        dct_pre(q, tk, z, zn);
        S[k * G] = z;
        if (kn != k) S[kn * G] = zn;
      }
    }
    __syncthreads();
  };
  if constexpr (!BL) {
    F::template run<G>(S, a.y.tw, t, false, [&](auto &v, int j, auto step) {
      gather<decltype(step)::value>(v, j, from_image);
    }, NoStore{});
    spectral();
    F::template run<G>(S, a.y.tw, t, true, [&](auto &v, int j, auto step) {
      gather<decltype(step)::value>(v, j, [&](int i) { return S[i * G]; });
    }, store_to(to_image));
  } else {
    dft<F, true, G>(S, a.y, t, false, [&](auto &v, int j, auto step) {
      gather<decltype(step)::value>(v, j, from_image);
    });
    spectral();
    int t2 = t;
    asm volatile("" : "+r"(t2));
    dft<F, true, G>(S, a.y, t2, true, [&](auto &v, int j, auto step) {
      gather<decltype(step)::value>(v, j, [&](int i) { return i < H ? S[i * G] : make_float2(0.f, 0.f); });
    });
    if (t < TP)
      for (int i = t; i < H; i += TP) to_image(i, S[i * G]);
  }
  if (kc == 0 || (kc == 1 && a.tight)) {
    acc = fct_block_sum(acc);
    if (threadIdx.x == 0) atomicAdd(&a.ctrl->rnorm2[fct_grid_slot(kc, c)], (double)acc);
  }
}

// Rows back: the correction e of G row pairs. The iterate is the sum of its corrections, each
// 1e-5 .. 1e-6 of the one before and kept as a part of its own: the first rounded to the channel's grid, and
// for rtol < 1e-6 the second to one too, or its Laplacian is only known to 3e-7 of a smooth field of
// 4096 x 4096 points. (A wider rtol does not need that, and the rounding could cost it a third cycle.)
template <class F, bool BL>
__global__ void __launch_bounds__(ceil_div(F::G_ROWS * F::TP, 32) * 32, blocks_per_sm(F::G_ROWS * F::TP))
fct_back_kernel(const __grid_constant__ FctArgs a, int kc) {
  griddep_enter();
  extern __shared__ float2 fct_sm[];
  constexpr int TP = F::TP, G = F::G_ROWS;
  const int c = blockIdx.y;
  const FctChannel ch = fct_block_channel(a, c, kc == 0 ? kFctFirst : kc);
  if (ch.skip) return;
  if (kc == 0 && blockIdx.x == 0 && threadIdx.x == 0) fct_record_goal(a, c, ch.lo, ch.sq);
  const int g = threadIdx.x / TP, t = g < G ? (int)threadIdx.x - g * TP : TP;
  float2 *S = fct_sm + (g < G ? g : 0) * F::template Layout<1>::SLOTS;
  const int W = a.W, H = a.H;
  const int ia = 2 * (blockIdx.x * G + g);
  const bool va = t < TP && ia < H, vb = t < TP && ia + 1 < H;
  const float *sa = a.spec + ((size_t)c * H + ia) * a.wp, *sb = sa + a.wp;
  auto packed = [&](int k) -> float2 {
    if (BL && k >= W) return make_float2(0.f, 0.f);
    const int kn = W - k;  // X[W] = 0
    const float ak = va ? __ldcg(sa + k) : 0.f, an = va && k > 0 ? __ldcg(sa + kn) : 0.f;
    const float bk = vb ? __ldcg(sb + k) : 0.f, bn = vb && k > 0 ? __ldcg(sb + kn) : 0.f;
    float2 z, zn;
    dct_pre(Quad{ak, an, bk, bn}, __ldg(a.x.th + k), z, zn);
    return z;
  };
  dft<F, BL, 1>(S, a.x, t, false, [&](auto &v, int j, auto step) { gather<decltype(step)::value>(v, j, packed); });
  constexpr float inv_len = 1.f / (float)F::LEN;
  float acc = 0.f;
  if (va) {
    const int half = (W + 1) / 2;
    // the third correction takes the place of its spectrum, row by row (which this block has read)
    const int pitch = kc > 1 ? a.wp : W;
    float *out = (kc == 0 ? a.uhi : kc == 1 ? a.ulo : a.spec) + (size_t)c * H * pitch;
    const bool round = kc == 0 || (kc == 1 && a.tight);
    const float grid = round ? fct_grid(a.ctrl->rnorm2[fct_grid_slot(kc, c)]) : 0.f;
    for (int m = t; m < half; m += TP) {
      const int j = 2 * m;
      const bool two = j + 1 < W;
      float2 z0 = S[m], z1 = two ? S[W - 1 - m] : z0;
      if (BL) {
        z0 = chirp_out(z0, __ldg(a.x.chirp + m), inv_len);
        if (two) z1 = chirp_out(z1, __ldg(a.x.chirp + W - 1 - m), inv_len);
      }
      const float2 e[2] = {make_float2(z0.y, z1.y), make_float2(z0.x, z1.x)};
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (r == 1 && !vb) break;
        float2 v = e[r];
        if (round) v = make_float2(__fsub_rn(__fadd_rn(v.x, grid), grid), __fsub_rn(__fadd_rn(v.y, grid), grid));
        acc += v.x;
        if (two) acc += v.y;
        st_pair(out + (size_t)(ia + r) * pitch, j, W, v);
      }
    }
  }
  acc = fct_block_sum(acc);
  if (threadIdx.x == 0) atomicAdd(&a.ctrl->sum_u[kc + 1][c], (double)acc);
}

// Bluestein: the FFT of the conjugate chirp exp(i pi t^2 / n), |t| < n, wrapped on LEN
// points (one block; side 0: x, 1: y).
template <class F>
__global__ void __launch_bounds__(ceil_div(F::TP, 32) * 32)
fct_chirp_kernel(const __grid_constant__ FctArgs a, int side) {
  griddep_enter();
  extern __shared__ float2 fct_sm[];
  const int n = side ? a.y.n : a.x.n, t = min((int)threadIdx.x, F::TP);
  const float2 *chirp = side ? a.y.chirp : a.x.chirp, *tw = side ? a.y.tw : a.x.tw;
  float2 *bhat = side ? a.y.bhat : a.x.bhat;
  F::template run<1>(fct_sm, tw, t, false, [&](auto &v, int j, auto step) {
    gather<decltype(step)::value>(v, j, [&](int i) -> float2 {
      const int q = i < n ? i : F::LEN - i;
      if (q >= n) return make_float2(0.f, 0.f);
      const float2 w = __ldg(chirp + q);
      return make_float2(w.x, -w.y);
    });
  }, store_to([&](int i, float2 v) { bhat[i] = v; }));
}

// The lengths by slice (one translation unit each): X(radices) for cosine transforms of
// that length, B(radices) for Bluestein's convolution.
#ifndef GDGS_FCT_LENGTHS
#define GDGS_FCT_LENGTHS_0(X, B) \
  X(8, 4, 1, 1) X(12, 12, 1, 1) X(15, 8, 3, 1) X(16, 16, 3, 1) X(15, 10, 10, 1) X(16, 15, 15, 1) B(15, 15, 4, 1) B(16, 16, 16, 2)
#define GDGS_FCT_LENGTHS_1(X, B) \
  X(12, 3, 1, 1) X(15, 10, 1, 1) X(16, 8, 3, 1) X(16, 10, 5, 1) X(16, 16, 6, 1) X(16, 16, 15, 1) B(15, 12, 6, 1)
#define GDGS_FCT_LENGTHS_2(X, B) \
  X(8, 5, 1, 1) X(16, 10, 1, 1) X(16, 5, 5, 1) X(15, 9, 6, 1) X(16, 10, 10, 1) X(16, 16, 16, 1) B(16, 16, 5, 1)
#define GDGS_FCT_LENGTHS_3(X, B) \
  X(16, 3, 1, 1) X(9, 6, 3, 1) X(12, 12, 3, 1) X(12, 12, 6, 1) X(15, 12, 9, 1) B(8, 4, 1, 1) B(16, 16, 6, 1)
#define GDGS_FCT_LENGTHS_4(X, B) \
  X(10, 5, 1, 1) X(15, 12, 1, 1) X(15, 6, 5, 1) X(15, 15, 4, 1) X(12, 12, 12, 1) B(16, 4, 1, 1) B(15, 15, 8, 1)
#define GDGS_FCT_LENGTHS_5(X, B) \
  X(9, 6, 1, 1) X(16, 12, 1, 1) X(15, 8, 4, 1) X(16, 15, 4, 1) X(15, 15, 8, 1) B(16, 6, 1, 1) B(15, 12, 12, 1)
#define GDGS_FCT_LENGTHS_6(X, B) \
  X(15, 4, 1, 1) X(8, 5, 5, 1) X(9, 9, 6, 1) X(12, 9, 9, 1) X(16, 15, 8, 1) B(16, 8, 1, 1) B(16, 16, 10, 1)
#define GDGS_FCT_LENGTHS_7(X, B) \
  X(16, 4, 1, 1) X(12, 6, 3, 1) X(10, 10, 5, 1) X(10, 10, 10, 1) X(16, 16, 8, 1) B(16, 10, 1, 1) B(16, 16, 12, 1)
#define GDGS_FCT_LENGTHS_8(X, B) \
  X(12, 6, 1, 1) X(16, 15, 1, 1) X(16, 8, 4, 1) X(16, 16, 4, 1) X(15, 12, 12, 1) B(8, 5, 5, 1) B(16, 15, 15, 1)
#define GDGS_FCT_LENGTHS_9(X, B) \
  X(16, 5, 1, 1) X(10, 5, 5, 1) X(15, 12, 3, 1) X(15, 12, 6, 1) X(15, 15, 10, 1) B(16, 15, 1, 1) B(16, 16, 16, 1)
#define GDGS_FCT_LENGTHS_10(X, B) \
  X(15, 6, 1, 1) X(16, 16, 1, 1) X(16, 12, 3, 1) X(16, 12, 6, 1) X(16, 12, 12, 1) B(16, 6, 3, 1) B(16, 16, 9, 2)
#define GDGS_FCT_LENGTHS_11(X, B) \
  X(16, 6, 1, 1) X(15, 6, 3, 1) X(15, 8, 5, 1) X(16, 15, 5, 1) X(16, 15, 10, 1) B(15, 8, 3, 1) B(16, 16, 10, 2)
#define GDGS_FCT_LENGTHS_12(X, B) \
  X(10, 10, 1, 1) X(16, 6, 3, 1) X(16, 8, 5, 1) X(16, 16, 5, 1) X(16, 16, 10, 1) B(12, 12, 3, 1) B(16, 15, 12, 2)
#define GDGS_FCT_LENGTHS_13(X, B) \
  X(12, 9, 1, 1) X(15, 5, 4, 1) X(12, 9, 6, 1) X(16, 9, 9, 1) X(15, 15, 12, 1) B(16, 8, 4, 1) B(16, 16, 12, 2)
#define GDGS_FCT_LENGTHS_14(X, B) \
  X(15, 8, 1, 1) X(16, 5, 4, 1) X(16, 15, 3, 1) X(15, 15, 6, 1) X(16, 15, 12, 1) B(16, 8, 5, 1) B(16, 12, 12, 3)
#define GDGS_FCT_LENGTHS_15(X, B) \
  X(16, 8, 1, 1) X(12, 9, 3, 1) X(15, 10, 5, 1) X(16, 15, 6, 1) X(16, 16, 12, 1) B(16, 16, 3, 1) B(16, 16, 15, 2)
#endif

// Defines this translation unit's slice of the lengths.
template <class F, bool BL>
constexpr FctEntry fct_entry() {
  return {F::LEN, BL ? 1 : 0, ceil_div(F::G_ROWS * F::TP, 32) * 32, F::G_ROWS,
          (int)sizeof(float2) * F::G_ROWS * F::template Layout<1>::SLOTS, ceil_div(F::G_COLS * F::TP, 32) * 32, F::G_COLS,
          (int)sizeof(float2) * F::G_COLS * F::template Layout<F::G_COLS>::SLOTS, ceil_div(F::TP, 32) * 32,
          (int)sizeof(float2) * F::template Layout<1>::SLOTS};
}

}  // namespace

}  // namespace gdgs

#define GDGS_FCT_KERNELS(A, B_, C_, D, BL)                                                    \
  fct_rows_kernel<Fft<A, B_, C_, D>, BL>, fct_cols_kernel<Fft<A, B_, C_, D>, BL>,             \
      fct_back_kernel<Fft<A, B_, C_, D>, BL>
#define GDGS_FCT_DIRECT(A, B_, C_, D) \
  {fct_entry<Fft<A, B_, C_, D>, false>(), GDGS_FCT_KERNELS(A, B_, C_, D, false), nullptr},
#define GDGS_FCT_CHIRP(A, B_, C_, D) \
  {fct_entry<Fft<A, B_, C_, D>, true>(), GDGS_FCT_KERNELS(A, B_, C_, D, true), fct_chirp_kernel<Fft<A, B_, C_, D>>},
#define GDGS_FCT_SLICE(N)                                                                        \
  namespace gdgs {                                                                               \
  const FctKernels *fct_slice##N(int *count) {                                                   \
    static const FctKernels e[] = {GDGS_FCT_LENGTHS_##N(GDGS_FCT_DIRECT, GDGS_FCT_CHIRP)};        \
    *count = (int)(sizeof(e) / sizeof(e[0]));                                                    \
    return e;                                                                                    \
  }                                                                                              \
  }
