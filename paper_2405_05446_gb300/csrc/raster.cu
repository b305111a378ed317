// Tile rasteriser of the per-Gaussian attribute (K5): the gradient (gx, gy per
// channel) or, in the paper-literal form, the Laplacian value per channel.
//
// One CTA per non-empty 16x16 tile. The tile's splats are already in front-to-back
// order (sort.cu); they are staged into shared memory and every pixel composites them as in
// Eq. gdgs2d (Eq. color with the gradient attribute):
//   G = exp(-k d^T conic d), a = min(alpha_max, alpha G), skip a < alpha_min,
//   acc += g a T, T -= a T, stop once T < t_min.
// Tiles no splat reaches are never launched (the field is sparse, Sec. 2.2).
//
// The splat is staged relative to the tile origin (stage_splat): its centre's
// (hi, lo) pair becomes a grid part that pixel centres subtract exactly and a
// remainder folded into the expanded exponent, so alpha keeps FP32 relative
// precision anywhere in the image. alpha = 2^(L - p2) with L = log2(opacity)
// (ex2.approx; k log2 e is folded into the conic at projection), taken for every splat
// whose ellipse reaches the warp's block.
//
// One CTA of 128 threads per tile; a warp holds an 8 x 8 pixel block and a lane two
// pixels of one column, 4 rows apart, whose arithmetic runs as packed FP32 pairs
// (add / mul / fma.f32x2: the same roundings as two scalar operations; a pair takes the
// FMA pipe two cycles but one issue slot, and the kernel is bound by issue). Operands that
// both pixels share sit in shared memory twice, side by side, so that a 16-byte broadcast
// load gives two ready pairs. Per splat and warp that is ~40 instructions for 64 pixels
// against ~33 for 32 pixels with a pixel per lane. There is no branch per pixel: a pixel
// below alpha_min gets weight 0, a stopped one transmittance 0.
//
// The warps of a tile work on their own: each walks the tile's list 32 splats at a time
// (a lane loads one and tests whether its ellipse reaches the warp's block), packs the ones
// that do into shared memory of its own in front-to-back order, composites them and stops
// when all its pixels have. Staging once per tile with barriers between the batches left
// the warps waiting for each other (ncu: 2.6 barrier stalls per issue, 62 % issue active).
//
// Measured on a GB300, the kernel alone, before (a pixel per lane, lists by the ellipse's
// bounding box, batches with barriers) and now: 1080p with 200k Gaussians 243 -> 195 us, 2160p
// with 1M 905 -> 737 us, 1237x711 with 300k and 4 channels 211 -> 181 us, 1080p Laplacian 231
// -> 174 us; 177M -> 130M warp-instructions at 1080p, 64 % issue active, the shared-memory
// pipe (seven 16-byte broadcasts per splat and warp) 61 % busy, DRAM 1 %.
#include "gdgs_internal.cuh"

namespace gdgs {

namespace {

constexpr int kRasterThreads = 128;
// Up to 16 tiles per SM (152) the warps are too few to hide the three loads that follow one
// another in a batch (index, splat, attribute), and the kernel loads ahead; above, the 8 to 34
// registers that takes cost more than they give. Without and with: 243x143 with 294k Gaussians
// 731 -> 534 us (144 tiles; a pixel per lane 659), 500x300 with 300k 348 -> 264 us (608 tiles),
// 1237x711 with 300k 180 -> 178 us (3510), the 1080p view 489 -> 494 us (8160), the 2160p one
// 1946 -> 2040 us (32400).
constexpr int kAheadTiles = 2432;

template <int Q, bool kAhead>
__global__ void __launch_bounds__(kRasterThreads) raster_kernel(RasterArgs a) {
  griddep_enter();
  constexpr int QP = (Q + 1) / 2;  // 16-byte slots of the doubled attribute
  // per warp, up to 32 splats, every value twice: (-h_x, -h_y), (A, B'), (a, C), (b, L) of
  // StagedSplat, then the attribute
  __shared__ float4 s_splat[kRasterThreads / 32][4 + QP][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned ntiles = a.use_active ? a.ctrl->n_active : (unsigned)a.T;
  if (blockIdx.x >= ntiles || a.ctrl->gave_up) return;  // no sorted list
  const int tile = a.use_active ? (int)a.active[blockIdx.x] : (int)blockIdx.x;
  const int tyi = tile / a.tiles_x, txi = tile - tyi * a.tiles_x;
  const int x0 = txi * kTile, y0 = tyi * kTile;
  const int bx = 8 * (warp & 1), by = 8 * (warp >> 1);  // the warp's block in the tile
  const int lx = bx + (lane & 7), ly = by + (lane >> 3);
  const int px = x0 + lx, py = y0 + ly;
  const bool in0 = px < a.W && py < a.H, in1 = px < a.W && py + 4 < a.H;
  const f32x2 fpx = pk(lx + 0.5f, lx + 0.5f), fpy = pk(ly + 0.5f, ly + 4.5f);
  const float x0f = (float)x0, y0f = (float)y0;
  const uint2 rg = tile_range(a.range, tile);
  const float amin = a.alpha_min, amax = a.alpha_max, tmin = a.t_min;
  const f32x2 minus1 = pk(-1.f, -1.f);
  float4(*S)[32] = s_splat[warp];

  f32x2 acc[Q];
#pragma unroll
  for (int q = 0; q < Q; ++q) acc[q] = pk(0.f, 0.f);
  float T0 = in0 ? 1.f : 0.f, T1 = in1 ? 1.f : 0.f;  // 0: stopped (or outside)

  // composites the n splats in shared memory
  auto composite = [&](int n) {
    for (int k = 0; k < n; ++k) {
      f32x2 X, Y;
      float t0, t1;
      staged_log2_alpha(&S[0][k], 32, fpx, fpy, X, Y, t0, t1);
      float al0 = fminf(amax, ex2_approx(t0)), al1 = fminf(amax, ex2_approx(t1));
      al0 = al0 >= amin ? al0 : 0.f;
      al1 = al1 >= amin ? al1 : 0.f;
      const f32x2 T = pk(T0, T1);
      const f32x2 w = mul2(pk(al0, al1), T);
#pragma unroll
      for (int v = 0; v < QP; ++v) {
        const ulonglong2 gg = *reinterpret_cast<const ulonglong2 *>(&S[4 + v][k]);
        acc[2 * v] = fma2(gg.x, w, acc[2 * v]);
        if (2 * v + 1 < Q) acc[2 * v + 1] = fma2(gg.y, w, acc[2 * v + 1]);
      }
      unpk(fma2(w, minus1, T), T0, T1);  // T (1 - a), reusing the weight (the backward replays this)
      T0 = T0 < tmin ? 0.f : T0;
      T1 = T1 < tmin ? 0.f : T1;
    }
  };
  // attribute of Gaussian g
  auto attribute = [&](uint32_t g, float (&gv)[2 * QP]) {
    const float *gp = a.grad + (size_t)g * Q;
    gv[2 * QP - 1] = 0.f;
    if (Q % 2 == 0 && a.grad_pairs) {  // 8-byte aligned rows: one 8-byte load per two floats
#pragma unroll
      for (int q = 0; q < Q; q += 2) {
        const float2 v2 = __ldg(reinterpret_cast<const float2 *>(gp + q));
        gv[q] = v2.x;
        gv[q + 1] = v2.y;
      }
    } else {
#pragma unroll
      for (int q = 0; q < Q; ++q) gv[q] = __ldg(gp + q);
    }
  };
  auto store = [&](const StagedSplat &st, const float (&gv)[2 * QP], int k) {
    store_pairs(st, &S[0][k], 32);
#pragma unroll
    for (int v = 0; v < QP; ++v) S[4 + v][k] = make_float4(gv[2 * v], gv[2 * v], gv[2 * v + 1], gv[2 * v + 1]);
  };

  if (kAhead) {
    // Three batches in flight: a batch's attributes are loaded while the one before it is
    // composited, its splats a batch earlier, their indices another batch earlier.
    uint32_t g1 = 0, g2 = 0;
    float4 sm1 = make_float4(0.f, 0.f, 0.f, 0.f), kc1 = sm1;
    if (rg.x + lane < rg.y) {
      g1 = a.pval[rg.x + lane];
      sm1 = a.smean[g1];
      kc1 = a.sconic[g1];
    }
    if (rg.x + 32 + lane < rg.y) g2 = a.pval[rg.x + 32 + lane];
    int n0 = 0;  // splats of the previous batch
    for (unsigned s = rg.x; s < rg.y; s += 32) {
      if (!__any_sync(0xffffffffu, T0 + T1 > 0.f)) break;
      const StagedSplat st = stage_splat(sm1, kc1, x0f, y0f);
      const bool in = s + lane < rg.y && reaches_block<8>(st, kc1, amin, by, bx);
      const unsigned ball = __ballot_sync(0xffffffffu, in);
      float gv[2 * QP] = {};
      if (in) attribute(g1, gv);
      g1 = g2;
      if (s + 32 + lane < rg.y) {
        sm1 = a.smean[g1];
        kc1 = a.sconic[g1];
      }
      if (s + 64 + lane < rg.y) g2 = a.pval[s + 64 + lane];
      composite(n0);
      __syncwarp();
      if (in) store(st, gv, __popc(ball & ((1u << lane) - 1u)));
      __syncwarp();
      n0 = __popc(ball);
    }
    composite(n0);  // (stopped pixels have T = 0: no weight)
  } else {
    for (unsigned s = rg.x; s < rg.y; s += 32) {
      if (!__any_sync(0xffffffffu, T0 + T1 > 0.f)) break;
      const unsigned j = s + lane;
      StagedSplat st;
      uint32_t g = 0;
      bool in = false;
      if (j < rg.y) {
        g = a.pval[j];
        const float4 kc = a.sconic[g];
        st = stage_splat(a.smean[g], kc, x0f, y0f);
        in = reaches_block<8>(st, kc, amin, by, bx);
      }
      const unsigned ball = __ballot_sync(0xffffffffu, in);
      if (in) {
        float gv[2 * QP];
        attribute(g, gv);
        store(st, gv, __popc(ball & ((1u << lane) - 1u)));
      }
      __syncwarp();
      composite(__popc(ball));
      __syncwarp();
    }
  }
  const size_t plane = (size_t)a.H * a.W;
  const size_t o = (size_t)py * a.W + px;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    float v0, v1;
    unpk(acc[q], v0, v1);
    if (in0) a.maps[q * plane + o] = v0;
    if (in1) a.maps[q * plane + o + (size_t)4 * a.W] = v1;
  }
}

template <int Q>
void launch_tiles(const RasterArgs &a, cudaStream_t st) {
  if (a.T <= kAheadTiles) launch_k(raster_kernel<Q, true>, a.T, kRasterThreads, 0, st, a);
  else launch_k(raster_kernel<Q, false>, a.T, kRasterThreads, 0, st, a);
}

}  // namespace

cudaError_t launch_raster(const RasterArgs &a_in, cudaStream_t st) {
  if (a_in.T == 0) return cudaSuccess;
  RasterArgs a = a_in;
  a.grad_pairs = (a.Q % 2 == 0 && (reinterpret_cast<uintptr_t>(a.grad) & 7u) == 0) ? 1 : 0;
  LaunchScope ls_("raster", st);
  switch (a.Q) {
    case 1: launch_tiles<1>(a, st); break;
    case 2: launch_tiles<2>(a, st); break;
    case 3: launch_tiles<3>(a, st); break;
    case 4: launch_tiles<4>(a, st); break;
    case 6: launch_tiles<6>(a, st); break;
    case 8: launch_tiles<8>(a, st); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace gdgs
