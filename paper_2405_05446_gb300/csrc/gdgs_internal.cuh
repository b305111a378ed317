// Internal declarations shared by the CUDA translation units of libgdgs.
// Not part of the ABI; include/gdgs.h is the public contract.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/gdgs.h"

namespace gdgs {

constexpr int kTile = GDGS_TILE;        // raster tile edge (pixels)
constexpr int kMaxCycles = 64;          // bound on V-cycles per solve
constexpr int kMaxLevels = 24;          // bound on multigrid levels
// Radix sorts (sort.cu): threads and keys per thread of a pass's tiles; threads
// per SM (four blocks of 64 registers); the histogram's threads; grids of a few
// resident blocks per SM (152).
constexpr int kSortThreadsPerSm = 1024;
constexpr int kDepthThreads = 256, kDepthItems = 8, kDepthTile = kDepthThreads * kDepthItems;
constexpr int kPairThreads = 256, kPairItems = 10, kPairTile = kPairThreads * kPairItems;
constexpr int kHistThreads = 512, kHistGrid = 304, kSortGrid = 1216, kEmitGrid = 912;
constexpr int kSortPasses = 5;  // of the depth sort; the pair sort has at most 4
constexpr int kDepthDigits = 256;
constexpr int kBinBlock = 256;  // Gaussians per block of the pair count and emission
constexpr uint32_t kInvalidKey = 0xFFFFFFFFu;

// Device control block at offset 0 of every workspace. Zeroed at the start of
// each call (except the fields after `persist_begin`, of which there are none:
// the coarse-solver cache lives in its own region).
struct Ctrl {
  int status;          // first device error (atomicCAS from GDGS_OK)
  int stopped;         // multigrid: convergence observed
  int cycles;          // multigrid: V-cycles behind the returned iterate
  int n_visible;       // Gaussians that survived projection
  unsigned long long n_pairs;  // (tile, splat) pairs requested (uncapped)
  unsigned n_active;   // tiles with at least one pair
  int gave_up;         // a sort's wait ran out: no order, no pairs (whatever status already holds)
  int max_cycles;
  int channels;
  int iter;            // cycle index when the cycle loop runs as a graph
  int direct;          // direct solve (cosine transforms): refinement cycles launched, 0 otherwise
  double rtol;
  double rnorm2[kMaxCycles + 1];             // ||rho - L u_k||^2, k = 0..
  double sum_u[kMaxCycles + 1][GDGS_MAX_CHANNELS];  // sum of u_k per channel
  double final_rnorm2;                       // residual of the returned iterate
  double mean_set[GDGS_MAX_CHANNELS];
  double rho_sum[GDGS_MAX_CHANNELS];         // sum and sum of squares of rho per channel
  double rho_sq[GDGS_MAX_CHANNELS];
  float rho_mean[GDGS_MAX_CHANNELS];         // the constant removed from rho (least squares)
  float escale[kMaxCycles + 1];              // cycle k solves for s_k e (a power of two)
  // channel split: every channel ran its own cycle loop (control block of its
  // own, off_sub); kf_c[c] is the cycle count of channel c's returned iterate
  int split;
  int kf_c[GDGS_MAX_CHANNELS];
};

// Direct solve: rnorm2[] holds each channel's ||residual||^2 after q = 1 .. cycles
// cycles, and (q = 0, written by the finalize pass) ||rho - mean||^2.
__host__ __device__ constexpr int fct_slot(int q, int c) { return 1 + GDGS_MAX_CHANNELS * q + c; }

// Diagnostics hooks around every kernel launch (diag.cu).
void diag_before(const char *name, cudaStream_t st);
void diag_after(cudaStream_t st);
bool diag_profiling();
void diag_set_capturing(bool on);  // launches on this thread are being captured into a graph
unsigned long long graph_kernel_count();  // kernels run by graph-launched cycle loops
// Programmatic dependent launch. Every kernel of the library begins with
// griddep_enter(), which waits until the kernel launched before it on the
// stream has completed and its writes are visible (griddepcontrol.wait).
// Kernels are launched with the programmatic-serialization attribute (below),
// so a dependent grid is launched as soon as every CTA of its predecessor has
// exited, overlapping the launch with the predecessor's completion, instead of
// after a full launch round trip. No kernel triggers its dependents early
// (griddepcontrol.launch_dependents): CTAs launched early would sit resident
// while they wait and take SM slots from kernels of other streams (measured:
// 583 against 721 mixed views/s when four streams serve views). The wait comes
// before any global access of every thread, so the order of all reads and
// writes is that of plain stream order, and a kernel completes only after its
// predecessor has.
__device__ __forceinline__ void griddep_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

bool pdl_enabled();  // GDGS_PDL=0 turns the attribute off (diag.cu)

// Launch with the programmatic-serialization attribute (when enabled). Errors
// are reported by the caller's cudaGetLastError, as for <<<>>> launches.
template <typename... K, typename... A>
inline void launch_k(void (*kern)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                     A &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, static_cast<A &&>(args)...);
}

struct LaunchScope {
  cudaStream_t st;
  LaunchScope(const char *name, cudaStream_t s) : st(s) { diag_before(name, s); }
  ~LaunchScope() { diag_after(st); }
};

__device__ __forceinline__ void set_status(Ctrl *c, int code) {
  atomicCAS(&c->status, GDGS_OK, code);
}
// A bounded wait ran out. The status may hold an earlier error (a capacity overflow, a non-finite
// parameter), so the kernels that follow go by a flag of its own: without a sorted list they
// would index with what an earlier call left in the workspace.
__device__ __forceinline__ void give_up(Ctrl *c) {
  set_status(c, GDGS_ERR_TIMEOUT);
  c->gave_up = 1;
}

// Geometry of one multigrid level. Level l has ceil(N0 / 2^l) cells per side;
// cell J covers fine pixels [J 2^l, min((J+1) 2^l, N0)), so only the last cell
// of a side may be narrower. Widths are normalised by 2^l (full cell = 1).
struct LevelGeom {
  int H, W;            // cells
  int shift;           // l
  int H0, W0;          // finest grid
  float lastx, lasty;  // normalised width of the last column / height of the last row
  float ex, ey;        // 2 / (1 + lastx), 2 / (1 + lasty): face factors next to them
  long long plane;     // floats per channel plane (H * W)
};

// ---------------------------------------------------------------- workspace plan
struct Plan {
  int64_t n;
  int C, W, H;
  int tiles_x, tiles_y, T;
  unsigned pair_cap;
  // offsets in bytes from the workspace base
  size_t off_ctrl;
  size_t off_smean, off_sconic, off_rect;              // projected splats [n]
  size_t off_dkey[2], off_dval[2];                     // depth sort [n]
  size_t off_dlo;                                      // depth sort secondary key [n]
  size_t off_hist, off_sort;                           // sorts: published words; counts and tickets (shared, make_plan)
  size_t off_blocksum;                                 // scan partials
  size_t off_gtiles;                                   // tiles per depth-ordered Gaussian
  size_t off_pkey[2], off_pval[2];                     // pairs [pair_cap]
  size_t off_range, off_active, off_mask;              // per tile
  size_t off_maps;                                     // [C][2][H][W]
  size_t off_dsplat;                                   // backward: [n][6] (shared, make_plan)
  size_t off_rho, off_uhi, off_ulo, off_e0, off_r[2];  // level 0 [C][H][W]
  size_t off_lu[kMaxLevels], off_lf[kMaxLevels];       // levels >= 1: down-pass u, f
  size_t off_luo[kMaxLevels];                          // levels >= 1: up-pass u (never in place)
  size_t off_coarse;                                   // tag + FP64 inverse
  size_t off_sub;                                      // per-channel control blocks [C]
  int levels;         // number of levels (finest = 0, coarsest = levels-1)
  int nc;             // unknowns on the coarsest level
  LevelGeom lv[kMaxLevels];
  size_t total;
};

bool make_plan(int64_t n, int C, int W, int H, const gdgs_raster_opts &ro,
               const gdgs_solver_opts &so, Plan *p);

constexpr size_t kCoarseTagBytes = 256;
struct CoarseTag {
  unsigned long long magic;
  int H0, W0, levels, Hc, Wc, nc;
  int version;
  int pad;
  unsigned long long hash;  // digest of the cached factor
};
constexpr int kMaxCoarse = 16 * 16;  // unknowns of the largest coarsest grid

// ---------------------------------------------------------------- launchers
// Each returns cudaSuccess or the launch error; all enqueue on `st`.
struct ProjectArgs {
  const float *mean, *scale, *quat, *opacity, *grad;
  int64_t n;
  int C;
  int Q;           // attribute floats per Gaussian
  float w2c[12];
  float fx, fy, cx, cy, znear;
  int W, H, tiles_x, tiles_y;
  uint32_t *sort_scratch;      // [sort_words], zeroed here for the sorts that follow (null: none does)
  unsigned sort_words;
  const gdgs_camera *cam_dev;  // when set, w2c .. znear are read from it on the device
  float alpha_min, dilation, exp_coef;
  // outputs (workspace)
  float4 *smean;   // mx_hi, my_hi, mx_lo, my_lo
  float4 *sconic;  // conic * exp_coef * log2(e) (a, 2b, c), opacity
  uint32_t *key;   // float bits of the depth's hi part, kInvalidKey when culled
  uint32_t *key_lo;  // 8-bit digit of the depth's lo part in units of ulp(hi) / 256
  uint2 *rect;     // x0 | x1 << 16, y0 | y1 << 16 (tiles, half open)
  // optional outputs
  float *o_mean2d, *o_cov2d, *o_depth;
  int32_t *o_rect;
  Ctrl *ctrl;
};
cudaError_t launch_project(const ProjectArgs &a, cudaStream_t st);

// Radix sorts of 32-bit keys with 32-bit values, stable (sort.cu). The scratch is zeroed by
// the projection; `state` holds what the tiles of two successive passes publish.
// (keys in tiles, digits of a pass; a sort of one pass has one set.)
size_t sort_state_words(long long keys, int tile, int digits, int passes);
struct SortState {
  uint32_t *tile, *sum, *prefix;  // [tiles][digits], [groups][digits] twice
};
struct SortScratch {
  uint32_t *bins;    // [passes][256]
  unsigned *ticket;  // [passes]
};

enum { kSortPlain, kSortLow, kSortRanges };

struct SortPass {
  const uint32_t *keys_in, *vals_in, *keys_next;
  uint32_t *keys_out, *vals_out;
  const unsigned long long *n_dev;
  unsigned cap;
  int shift;
  const uint32_t *bins;
  unsigned *ticket;
  SortState state, state_next;  // this pass's; the next one's, cleared here (tile null: none)
  Ctrl *ctrl;
  uint2 *range;
  uint32_t *active;
  uint8_t *tile_mask;
};

// The Gaussians by depth: the primary keys' 32 bits, ties by the low 8 bits of key_lo, then
// by index; the indices in order end up in val[1]. Also clears the tile ranges and mask.
struct DepthSort {
  uint32_t *key[2], *val[2];
  const uint32_t *key_lo;
  unsigned n;
  uint32_t *state;
  SortScratch scratch;
  uint2 *range;
  uint8_t *tile_mask;
  int T;
  Ctrl *ctrl;
};
cudaError_t sort_depth(const DepthSort &s, cudaStream_t st);

// The pairs by tile: the Gaussians in order end up in val[pair_passes(T) & 1], each tile's
// pairs in range (tile_range), the tiles that have any in active (ctrl->n_active of them,
// in any order) and as 1 in tile_mask.
struct PairSort {
  uint32_t *key[2], *val[2];
  const unsigned long long *n_dev;
  unsigned cap;
  int T;
  uint32_t *state;
  SortScratch scratch;
  uint2 *range;
  uint32_t *active;
  uint8_t *tile_mask;
  Ctrl *ctrl;
};
cudaError_t sort_pairs(const PairSort &s, cudaStream_t st);

inline int tile_bits(int T) {
  int b = 1;
  while ((1 << b) < T) ++b;
  return b;
}
inline int pair_passes(int T) { return (tile_bits(T) + 7) / 8; }
inline int pair_digit(int T) { return (tile_bits(T) + pair_passes(T) - 1) / pair_passes(T); }
__host__ __device__ inline int pair_digits(int digit) { return 1 << (digit < 5 ? 5 : digit); }  // (the passes have 5 bits or more)
// Both sorts' digit counts and tickets: depth counts [kSortPasses][256], tickets [8] and [8], pair
// counts [pair_passes][256] (the last pass's digits only).
inline unsigned sort_words(int T) {
  return kSortPasses * 256 + 16 + (pair_passes(T) - 1) * 256 + pair_digits(pair_digit(T));
}
inline SortScratch depth_scratch(uint32_t *w) { return {w, w + kSortPasses * 256}; }
inline SortScratch pair_scratch(uint32_t *w) { return {w + kSortPasses * 256 + 16, w + kSortPasses * 256 + 8}; }

// A tile's pairs: the sort leaves (~start, end), zero where there are none.
__device__ __forceinline__ uint2 tile_range(const uint2 *range, int tile) {
  const uint2 r = range[tile];
  return r.y ? make_uint2(~r.x, r.y) : make_uint2(0u, 0u);
}

struct BinArgs {
  const uint32_t *order;   // Gaussian indices in depth order [n]
  const uint2 *rect;
  const float4 *smean, *sconic;  // projected splats (ellipse test of each tile of the rect)
  float alpha_min;
  int64_t n;
  int tiles_x, T;
  unsigned pair_cap;
  unsigned long long *blocksum;  // [ceil(n / kBinBlock) + 1]
  uint32_t *tiles;         // [n] tiles each depth-ordered Gaussian reaches (count -> emit)
  uint32_t *pkey, *pval;   // emitted pairs
  uint32_t *bins, *sort_state;  // the pair sort's digit counts and published words
  Ctrl *ctrl;
  SortState state;         // set by launch_emit_pairs, with the sort's passes
  int passes, digit;
};
cudaError_t launch_emit_pairs(const BinArgs &a, cudaStream_t st);

// A projected splat staged for the 16x16 tile whose origin is (x0, y0), as the
// forward and the backward rasteriser both evaluate it (the backward replays
// the forward's arithmetic exactly). The centre relative to the tile origin is
// split into a part h on a 2^-12 pixel grid and a remainder l (|l| <= 2^-13 px,
// carried from the projection's float-float centre): a pixel centre minus h is
// exact in FP32, and l enters through the linear and constant terms of the
// expanded exponent, so no offset is rounded at the tile's scale. With
// X = px - h, Y = py - h_y and the stored conic (A, B', C) (k log2 e folded in):
//   p2 = A dx^2 + B' dx dy + C dy^2, dx = X - l_x, dy = Y - l_y,
//      = X (A X + B' Y + a) + Y (C Y + b) + c0,
//   a = -(2 A l_x + B' l_y), b = -(B' l_x + 2 C l_y), c0 = A l_x^2 + B' l_x l_y + C l_y^2,
// and alpha = opacity 2^-p2 = 2^(L - (p2 - c0)) with L = log2(opacity) - c0.
struct StagedSplat {
  float4 geo;   // h_x, h_y, A, B'
  float4 geo2;  // C, L, a, b
  float lx, ly;
};

__device__ __forceinline__ float2 split_tile_offset(float hi, float lo, float origin) {
  // hi - origin exactly as s + e (TwoSum), then s = h + (s - h) with h on the grid
  const float s = __fadd_rn(hi, -origin), bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(-origin, bb));
  const float h = __fmul_rn(rintf(__fmul_rn(s, 4096.f)), 1.f / 4096.f);
  return make_float2(h, __fadd_rn(__fsub_rn(s, h), __fadd_rn(e, lo)));  // s - h is exact
}

// smean = (x_hi, y_hi, x_lo, y_lo), sconic = (A, B', C, opacity)
__device__ __forceinline__ StagedSplat stage_splat(float4 m, float4 k, float x0f, float y0f) {
  const float2 ox = split_tile_offset(m.x, m.z, x0f), oy = split_tile_offset(m.y, m.w, y0f);
  const float lx = ox.y, ly = oy.y;
  const float a = -fmaf(2.f * k.x, lx, k.y * ly), b = -fmaf(k.y, lx, 2.f * k.z * ly);
  const float c0 = fmaf(k.x * lx, lx, fmaf(k.y * lx, ly, k.z * ly * ly));
  StagedSplat st;
  st.geo = make_float4(ox.x, oy.x, k.x, k.y);
  st.geo2 = make_float4(k.z, log2f(k.w) - c0, a, b);
  st.lx = lx;
  st.ly = ly;
  return st;
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed FP32 pairs.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpk(f32x2 v, float &a, float &b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// A splat staged for the packed rasterisers, every value twice (both pixels of a lane):
// (-h_x, -h_y), (A, B'), (a, C), (b, L).
__device__ __forceinline__ void store_pairs(const StagedSplat &st, float4 *s, int stride) {
  s[0] = make_float4(-st.geo.x, -st.geo.x, -st.geo.y, -st.geo.y);
  s[stride] = make_float4(st.geo.z, st.geo.z, st.geo.w, st.geo.w);
  s[2 * stride] = make_float4(st.geo2.z, st.geo2.z, st.geo2.x, st.geo2.x);
  s[3 * stride] = make_float4(st.geo2.w, st.geo2.w, st.geo2.y, st.geo2.y);
}

// log2 of alpha (before its clamp) at a lane's two pixels, L - p2 + c0 with the expanded
// exponent X (A X + (B' Y + a)) + Y (C Y + b); X and Y are the offsets to h.
__device__ __forceinline__ void staged_log2_alpha(const float4 *s, int stride, f32x2 fpx, f32x2 fpy, f32x2 &X, f32x2 &Y,
                                                  float &t0, float &t1) {
  const ulonglong2 h = *reinterpret_cast<const ulonglong2 *>(s);
  const ulonglong2 ab = *reinterpret_cast<const ulonglong2 *>(s + stride);
  const ulonglong2 lc = *reinterpret_cast<const ulonglong2 *>(s + 2 * stride);
  const ulonglong2 bl = *reinterpret_cast<const ulonglong2 *>(s + 3 * stride);
  X = add2(fpx, h.x);
  Y = add2(fpy, h.y);
  const f32x2 u = fma2(ab.x, X, fma2(ab.y, Y, lc.x));
  const f32x2 p = fma2(X, u, mul2(Y, fma2(lc.y, Y, bl.x)));
  unpk(fma2(p, pk(-1.f, -1.f), bl.y), t0, t1);
}

// Which splats reach a block of a 16 x 16 tile (the rasterisers' warps hold 8 x 8 pixels):
// those whose ellipse p2 <= log2(opacity / alpha_min) + 1e-3 (the exponent cut of the
// composite), widened like the binning's cut (0.1 % + 0.01), meets the block's pixel
// centres. The ellipse cut by a band of rows is convex, so its x-extent is one interval:
// its right end is the ellipse's rightmost point if that lies in the band, else the larger
// of the boundary's values at the band's two ends (the left end likewise). Against the
// ellipse's bounding box 16-19 % fewer (splat, 4 x 8 block) pairs remain, exactly those with
// a contributing pixel (120k pairs sampled from views of 1237x711 to 3840x2160). D = 4AC - B^2 is
// computed without the cancellation error of the plain difference, which elongated splats
// need.
struct Reach {
  float cx, cy, hx, hy, bx, cutA, dA, oy;
  bool all;  // degenerate: reaches every block
};
__device__ __forceinline__ Reach splat_reach(const StagedSplat &st, float4 k, float amin) {
  Reach r;
  const float A = k.x, B = k.y, C = k.z;
  const float lim = (log2f(k.w / amin) + 1e-3f) * 1.001f + 0.01f;
  const float bb = __fmul_rn(B, B);
  const float D = __fadd_rn(fmaf(4.f * A, C, -bb), fmaf(-B, B, bb));
  r.all = !(lim > 0.f) || !(D > 0.f) || !(A > 0.f) || !(C > 0.f);
  r.hy = sqrtf(lim * 4.f * A / D) * 1.0001f + 1e-3f;
  r.hx = sqrtf(lim * 4.f * C / D) * 1.0001f + 1e-3f;
  r.cx = st.geo.x + st.lx;
  r.cy = st.geo.y + st.ly;
  r.bx = B / (2.f * A);
  r.cutA = lim / A;
  r.dA = D / (4.f * A * A);
  r.oy = B / (2.f * C) * r.hx;  // rightmost point at cy - oy, leftmost at cy + oy
  return r;
}
// The x-extent [*xl, *xr] of the ellipse in the band of pixel centres [y0, y1]; false: none.
__device__ __forceinline__ bool band_extent(const Reach &r, float y0, float y1, float *xl, float *xr) {
  const float ya = fmaxf(y0, r.cy - r.hy) - r.cy, yb = fminf(y1, r.cy + r.hy) - r.cy;
  const float wa = sqrtf(fmaxf(r.cutA - r.dA * ya * ya, 0.f)), wb = sqrtf(fmaxf(r.cutA - r.dA * yb * yb, 0.f));
  const float ca = r.cx - r.bx * ya, cb = r.cx - r.bx * yb;
  *xr = (-r.oy >= ya && -r.oy <= yb) ? r.cx + r.hx : fmaxf(ca + wa, cb + wb) + 1e-3f;
  *xl = (r.oy >= ya && r.oy <= yb) ? r.cx - r.hx : fminf(ca - wa, cb - wb) - 1e-3f;
  return ya <= yb;
}

// Whether the splat reaches the block of BH rows x 8 columns at (row, col) of its tile.
template <int BH>
__device__ __forceinline__ bool reaches_block(const StagedSplat &st, float4 k, float amin, int row, int col) {
  const Reach r = splat_reach(st, k, amin);
  float xl, xr;
  const bool band = band_extent(r, row + 0.5f, row + (BH - 0.5f), &xl, &xr);
  return r.all || (band && xl <= col + 7.5f && xr >= col + 0.5f);
}

struct RasterArgs {
  const float4 *smean, *sconic;
  const float *grad;
  const uint32_t *pval;     // Gaussian index of each sorted pair
  const uint2 *range;       // [T]
  const uint32_t *active;   // [T] active tile ids (when use_active)
  int use_active;           // 1: only active tiles (count in ctrl->n_active)
  int Q, W, H, tiles_x, T;  // Q attribute floats per Gaussian = output planes
  int grad_pairs;           // set by launch_raster: Q even and grad 8-byte aligned
  float alpha_min, alpha_max, t_min;
  float *maps;              // [Q][H][W]
  Ctrl *ctrl;
};
cudaError_t launch_raster(const RasterArgs &a, cudaStream_t st);

struct PoissonArgs {
  const float *maps;        // [C][2][H][W], or [C][H][W] when input_is_rho
  int input_is_rho;         // the field rho itself instead of gradient maps
  float threshold;          // hard threshold on rho (0: none)
  const uint8_t *mask;      // [tiles_y][tiles_x] or null
  int C, H, W, tiles_x;
  float mean[GDGS_MAX_CHANNELS];
  float *image;             // [C][H][W]
  int nu1, nu2, max_cycles;
  float rtol;
  float omega;              // smoother over-relaxation
  int storage;              // GDGS_STORAGE_*: multigrid corrections and coarse right-hand sides
  int coarse_max_dim;
  const Plan *plan;
  char *ws;
  Ctrl *ctrl;
};
cudaError_t run_poisson(const PoissonArgs &a, cudaStream_t st);

// ---------------------------------------------------------------- backward
struct DivAdjArgs {
  const float *rbar;     // d loss / d rho [C][H][W]
  const float *rho_fwd;  // the forward's thresholded rho (null: no threshold)
  const uint8_t *mask;   // forward tile mask (null: none)
  int input_is_rho;      // Laplacian attribute: maps are rho itself
  int C, H, W, tiles_x;
  float *mbar;           // d loss / d maps [Q][H][W]
};
cudaError_t launch_divergence_adjoint(const DivAdjArgs &a, cudaStream_t st);

struct RasterBwdArgs {
  const float4 *smean, *sconic;
  const float *attr;        // per-Gaussian attribute [n][Q]
  const uint32_t *pval;     // the forward's sorted pairs
  const uint2 *range;
  const uint32_t *active;
  int Q, W, H, tiles_x, T;
  float alpha_min, alpha_max, t_min;
  const float *mbar;        // d loss / d maps [Q][H][W]
  double *dsplat;           // [n][6]: centre x, y; moments xx, xy, yy of w (raster_backward_kernel); opacity (accumulated)
  float *dattr;             // [n][Q] (accumulated)
  Ctrl *ctrl;
};
cudaError_t launch_raster_backward(const RasterBwdArgs &a, cudaStream_t st);

struct ProjBwdArgs {
  const float *mean, *scale, *quat;
  int64_t n;
  float w2c[12];
  float fx, fy;
  float dilation, exp_coef;
  const double *dsplat;
  float *d_mean, *d_scale, *d_quat, *d_opacity;
};
cudaError_t launch_project_backward(const ProjBwdArgs &a, cudaStream_t st);

}  // namespace gdgs
