// Binning of splats into 16x16 tiles in front-to-back order (K2-K4).
//
// The composite of Eq. color / Eq. gdgs2d visits splats "sorted from the view
// direction". The path orders them in two stable sorts instead of one wide key:
//   1. sort the Gaussians by their camera depth, held as a float-float pair
//      (hi, lo): one pass over an 8-bit digit of lo in units of ulp(hi) / 256,
//      then four passes over the float bits of hi (positive floats sort as
//      unsigned integers). Pairs with equal hi are thereby ordered by lo, which
//      resolves the depth to 2^-31 relative instead of float32's 2^-24 (N items);
//   2. walk them in that order, emit one (tile, Gaussian) pair per touched tile,
//      so pairs come out depth-ordered;
//   3. stable-sort the pairs by tile id only (ceil(log2 T) bits, 2 passes at
//      1080p). Stability keeps depth order inside each tile, ties by index.
// Compared with a 64-bit (tile | depth) key this sorts 13 instead of 45 bits per
// pair and moves 8 instead of 12 bytes per pair and pass.
//
// Each sort is one histogram kernel (the digit counts of every pass at once) and one
// kernel per 8-bit pass that reads and writes every element once: a block ranks a tile of
// keys, gets the counts of the tiles before it by looking back through their published
// words (decoupled look-back: Merrill and Garland 2016; one pass per digit: Adinets and
// Merrill 2022), reorders the tile in shared memory and writes runs of equal digits. The
// last pass of the pair sort writes no keys: it leaves the tile ranges itself.
#include <algorithm>

#include "gdgs_internal.cuh"

namespace gdgs {

namespace {

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ unsigned item_count(const unsigned long long *n_dev, unsigned cap) {
  if (!n_dev) return cap;
  const unsigned long long n = *n_dev;
  return n < cap ? (unsigned)n : cap;
}

// Words that a pass's tiles leave for the tiles after them, one per digit:
//   per tile        1 + the number of its keys (0: not there yet);
//   per 16 tiles    the sum of their counts, and in the top bits how many of them it has;
//   per 16 tiles    kPrefix | the keys of smaller digits and those of this digit in all tiles
//                   up to the group's last (31 bits: there are at most 2^31 - 1 pairs).
// A tile adds its own group's earlier tiles and then walks back group by group to the first
// prefix. Walking back tile by tile instead read about 100 words a digit (several hundred
// tiles are in flight): 140 us for a pass over 16.4M pairs.
constexpr uint32_t kPrefix = 0x80000000u;
constexpr int kGroup = 16, kGroupBits = 24;
constexpr int kLookBack = 4;             // groups read at a time
constexpr int kLookBackLimit = 1 << 19;  // polls before the wait gives up (about a second)

__device__ __forceinline__ uint32_t ld_status(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_status(uint32_t *p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Exclusive scan of one value per digit, held by threads 0 .. 255 of a block.
template <int THREADS>
__device__ __forceinline__ unsigned scan_digits(unsigned v) {
  __shared__ unsigned wt[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31 && w < 8) wt[w] = x;
  __syncthreads();
  unsigned before = 0;
#pragma unroll
  for (int k = 0; k < 7; ++k)
    if (k < w) before += wt[k];
  return x - v + before;
}

// Clears what the tiles of a pass publish, by threads tid of nt.
__device__ __forceinline__ void clear_state(const SortState &s, unsigned tiles, unsigned digits, unsigned tid, unsigned nt) {
  const unsigned groups = (tiles + kGroup - 1) / kGroup;
  for (unsigned t = tid; t < tiles * digits; t += nt) s.tile[t] = 0u;
  for (unsigned t = tid; t < groups * digits; t += nt) s.sum[t] = s.prefix[t] = 0u;
}

// Digit counts of all passes of the depth sort (bins zeroed before), the cleared state of its
// first pass, and the cleared tile ranges and mask of the pair sort that follows.
__global__ void __launch_bounds__(kHistThreads) depth_hist_kernel(DepthSort a, SortState state) {
  griddep_enter();
  __shared__ unsigned sh[kSortPasses][256];
  const unsigned tid = blockIdx.x * kHistThreads + threadIdx.x, nt = gridDim.x * kHistThreads;
  for (int t = threadIdx.x; t < kSortPasses * 256; t += kHistThreads) (&sh[0][0])[t] = 0u;
  clear_state(state, (a.n + kDepthTile - 1) / kDepthTile, kDepthDigits, tid, nt);
  for (unsigned t = tid; t < (unsigned)a.T; t += nt) {
    a.range[t] = make_uint2(0u, 0u);
    a.tile_mask[t] = 0;
  }
  __syncthreads();
  for (unsigned i = tid; i < a.n; i += nt) {
    const uint32_t k = a.key[0][i];
    atomicAdd(&sh[0][a.key_lo[i] & 255u], 1u);
#pragma unroll
    for (int p = 1; p < kSortPasses; ++p) atomicAdd(&sh[p][(k >> (8 * p - 8)) & 255u], 1u);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < kSortPasses * 256; t += kHistThreads) {
    const unsigned c = (&sh[0][0])[t];
    if (c) atomicAdd(&a.scratch.bins[t], c);
  }
}

// One stable pass over 8 bits (or fewer) of the keys. Blocks draw tiles in order from a
// ticket, so a tile waits only for tiles whose blocks already run; the waits are bounded.
// What bounds it: the latency of a tile's chain (load, rank, look back, write) at half the
// issue rate; the traffic is 16 bytes a pair, 40 us at 16.4M. Tiles of 2560 pairs with four
// blocks an SM (64 registers without spills) were the fastest of 1536 .. 8192; ranking by
// votes over the digit's bits (32 instructions) came out equal, __match_any_sync 20 % slower.
// The seven passes of a 3840x2160 view (1M Gaussians, 16.4M pairs) 333 us, of 1920x1080 (200k,
// 1.3M) 88 us, launch gaps included; block histogram, scan and scatter kernels for each pass
// and a pass for the tile ranges took 735 and 196 us.
// kKind: kSortPlain; kSortLow: ranked by the secondary keys, values are the indices and the
// keys written are the primary ones; kSortRanges: the last pass over the pairs, whose output
// is the values and each tile's range.
template <int THREADS, int ITEMS, int BITS, int kKind>
__global__ void __launch_bounds__(THREADS, kSortThreadsPerSm / THREADS) sort_pass_kernel(SortPass a) {
  griddep_enter();
  constexpr int kWarps = THREADS / 32, kKeys = THREADS * ITEMS;
  constexpr unsigned kMask = (1u << BITS) - 1u;
  constexpr int kDigits = 1 << BITS;
  static_assert(THREADS >= 256 && THREADS % 32 == 0, "a thread per digit");
  static_assert(ITEMS <= 32, "the list of run heads takes the counters' place, 16 bits a key");
  extern __shared__ uint32_t sort_sm[];
  uint32_t *const sk = sort_sm, *const sv = sk + kKeys;
  uint2 *const wcnt = reinterpret_cast<uint2 *>(sv + kKeys);  // per warp and digit
  __shared__ unsigned s_tile, s_heads, s_first[256], s_out[256];
  const unsigned n = item_count(a.n_dev, a.cap), tiles = (n + kKeys - 1) / kKeys;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  uint2 *const row = wcnt + w * 256;
  uint16_t *const head = reinterpret_cast<uint16_t *>(wcnt);
  const unsigned lt = lanemask_lt();
  // (one thread looks: a block leaves as a whole, also when another one gives up meanwhile)
  if (tid == 0) s_tile = a.ctrl->gave_up ? ~0u : atomicAdd(a.ticket, 1u);
  for (;;) {
    for (int t = tid; t < kWarps * 256; t += THREADS) wcnt[t] = make_uint2(0u, 0u);
    __syncthreads();
    const unsigned tile = s_tile;
    if (tile >= tiles) break;
    const unsigned first = tile * (unsigned)kKeys, cnt = min(n - first, (unsigned)kKeys);
    const unsigned group = tile / kGroup, member = tile % kGroup;
    if (a.state_next.tile && tid < kDigits) {
      a.state_next.tile[(size_t)tile * kDigits + tid] = 0u;
      if (member == 0) a.state_next.sum[group * kDigits + tid] = a.state_next.prefix[group * kDigits + tid] = 0u;
    }
    // a warp's keys are consecutive: index = (warp, item, lane)
    const unsigned at = w * (32 * ITEMS) + lane;
    uint32_t key[ITEMS];
    unsigned pos[(ITEMS + 1) / 2] = {};  // two 16-bit ranks a word
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) key[r] = at + 32 * r < cnt ? a.keys_in[first + at + 32 * r] : 0u;
    // rank among the warp's keys: the lanes of a digit meet in its word's mask
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const bool in = at + 32 * r < cnt;
      uint2 *const slot = row + ((key[r] >> a.shift) & kMask);
      if (in) atomicOr(&slot->y, 1u << lane);
      __syncwarp();
      const uint2 v = *slot;  // (keys of earlier items, lanes of this one)
      const unsigned mine = __popc(v.y & lt);
      __syncwarp();
      if (in && mine == 0) *slot = make_uint2(v.x + __popc(v.y), 0u);
      __syncwarp();
      pos[r / 2] |= (v.x + mine) << (16 * (r & 1));
    }
    uint32_t val[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      if (kKind == kSortLow) val[r] = first + at + 32 * r;
      else val[r] = at + 32 * r < cnt ? a.vals_in[first + at + 32 * r] : 0u;
    }
    __syncthreads();
    unsigned c = 0;
    if (tid < 256) {
#pragma unroll
      for (int k = 0; k < kWarps; ++k) {
        const unsigned x = wcnt[k * 256 + tid].x;
        wcnt[k * 256 + tid].x = c;
        c += x;
      }
      if (tid < kDigits) {
        st_status(&a.state.tile[(size_t)tile * kDigits + tid], 1u + c);
        atomicAdd(&a.state.sum[group * kDigits + tid], (1u << kGroupBits) + c);
      }
    }
    const unsigned ex = scan_digits<THREADS>(c);
    unsigned base = 0;
    if (group == 0) {  // uniform: the first group starts at the digits' places
      __syncthreads();
      base = scan_digits<THREADS>(tid < kDigits ? a.bins[tid] : 0u);
    }
    if (tid < 256) s_first[tid] = ex;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      if (at + 32 * r < cnt) {
        const unsigned d = (key[r] >> a.shift) & kMask;
        const unsigned q = s_first[d] + row[d].x + ((pos[r / 2] >> (16 * (r & 1))) & 0xffffu);
        sk[q] = key[r];
        sv[q] = val[r];
      }
    }
    if (tid <= kMask) {
      int polls = 0;
      for (bool done = false; !done;) {  // the earlier tiles of the group
        uint32_t s[kGroup - 1];
#pragma unroll
        for (int k = 0; k < kGroup - 1; ++k)
          s[k] = k < (int)member ? ld_status(&a.state.tile[(size_t)(tile - 1 - k) * kDigits + tid]) : 1u;
        unsigned sum = 0;
        done = true;
#pragma unroll
        for (int k = 0; k < kGroup - 1; ++k) {
          done = done && s[k] != 0u;
          sum += s[k] - 1u;
        }
        if (!done && ++polls > kLookBackLimit) {  // give up; the guard below keeps writes in bounds
          give_up(a.ctrl);
          done = true;
        }
        if (done) base += sum;
        else __nanosleep(64);
      }
      int g = (int)group - 1;
      for (bool done = g < 0; !done;) {
        uint32_t pre[kLookBack], sum[kLookBack];
#pragma unroll
        for (int k = 0; k < kLookBack; ++k) {
          pre[k] = g - k >= 0 ? ld_status(&a.state.prefix[(g - k) * kDigits + tid]) : 0u;
          // (group 0: its prefix, which has the smaller digits' keys)
          sum[k] = g - k > 0 ? ld_status(&a.state.sum[(g - k) * kDigits + tid]) : 0u;
        }
        bool go = true;
#pragma unroll
        for (int k = 0; k < kLookBack; ++k) {
          if (go && pre[k]) {
            base += pre[k] & ~kPrefix;
            done = true;
          } else if (go && sum[k] >> kGroupBits == kGroup) {
            base += sum[k] & ((1u << kGroupBits) - 1u);
            --g;
          } else {
            go = false;
          }
          go = go && !done;
        }
        if (!done && ++polls > kLookBackLimit) {
          give_up(a.ctrl);
          done = true;
        }
        if (!go && !done) __nanosleep(64);
      }
      if (member == kGroup - 1) st_status(&a.state.prefix[group * kDigits + tid], kPrefix | ((base + c) & ~kPrefix));
      s_out[tid] = base - ex;
    }
    if (kKind == kSortRanges && tid == 0) s_heads = 0;
    __syncthreads();
    if (tid == 0) s_tile = atomicAdd(a.ticket, 1u);
#pragma unroll 4
    for (int r = 0; r < ITEMS; ++r) {
      const unsigned i = tid + r * THREADS;
      if (i < cnt) {
        const uint32_t k = sk[i], v = sv[i];
        const unsigned q = s_out[(k >> a.shift) & kMask] + i;
        if (q < n) {
          a.vals_out[q] = v;
          if (kKind == kSortPlain) a.keys_out[q] = k;
          if (kKind == kSortLow) a.keys_out[q] = a.keys_next[v];
          if (kKind == kSortRanges) {
            // Runs of one tile are consecutive here (the earlier passes sorted the lower
            // bits). Their ends go into the tile's range by a maximum, their heads are listed.
            if (i + 1 == cnt || sk[i + 1] != k) atomicMax(&a.range[k].y, q + 1);
            if (i == 0 || sk[i - 1] != k) head[atomicAdd(&s_heads, 1u)] = (uint16_t)i;
          }
        }
      }
    }
    if (kKind == kSortRanges) {
      // The heads: ~start by a maximum (0: none yet). The block that finds none lists the
      // tile as active (in any order). All at once: an atomic's answer takes about 1 us.
      __syncthreads();
      const unsigned heads = s_heads;
      for (unsigned h0 = w * 32; h0 < heads; h0 += THREADS) {
        const unsigned h = h0 + lane;
        uint32_t k = 0u;
        bool fresh = false;
        if (h < heads) {
          const unsigned i = head[h];
          k = sk[i];
          fresh = atomicMax(&a.range[k].x, ~(s_out[(k >> a.shift) & kMask] + i)) == 0u;
        }
        const unsigned ball = __ballot_sync(0xffffffffu, fresh);
        unsigned at0 = 0;
        if (lane == 0 && ball) at0 = atomicAdd(&a.ctrl->n_active, __popc(ball));
        at0 = __shfl_sync(0xffffffffu, at0, 0);
        if (fresh) {
          a.active[at0 + __popc(ball & lt)] = k;
          a.tile_mask[k] = 1;
        }
      }
      __syncthreads();  // before the counters are cleared for the next tile
    }
  }
}

// ---------------------------------------------------------------- pair emission

__device__ __forceinline__ unsigned rect_tiles(uint2 r) {
  const unsigned x0 = r.x & 0xffffu, x1 = r.x >> 16, y0 = r.y & 0xffffu, y1 = r.y >> 16;
  return (x1 - x0) * (y1 - y0);
}

// Block-wide exclusive scan of 64-bit values for 256 threads.
__device__ unsigned long long block_exclusive_scan(unsigned long long v, unsigned long long *total) {
  __shared__ unsigned long long wt[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wt[w] = x;
  __syncthreads();
  unsigned long long before = 0, all = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    if (k < w) before += wt[k];
    all += wt[k];
  }
  __syncthreads();
  *total = all;
  return x - v + before;
}

// Sum of tile counts per block of kBinBlock depth-ordered Gaussians.
// The tiles a splat reaches: per row of tiles of its footprint box, the run of
// tiles whose box of pixel centres meets the ellipse p <= cut', where p = A dx^2
// + B dx dy + C dy^2 is the splat's exponent (conic with k log2 e folded in) and
// cut' the rasteriser's cut log2(opacity / alpha_min) + 1e-3 with a further
// 0.1 % + 0.01 of margin, so a dropped tile never holds a pixel where
// a >= alpha_min. The ellipse cut by a band of rows is convex, so its x-extent
// is one interval: on the right, the ellipse's rightmost point if that point's
// y lies in the band, else the larger value of the (concave) boundary function
// x = mx - B/(2A) dy + sqrt(cut'/A - D/(4A^2) dy^2), D = 4AC - B^2, at the
// band's ends; the left side likewise. A tile meets the ellipse iff its
// pixel-centre interval meets that extent.
struct Footprint {
  float mx, my, bx, cutA, dA, ry, rx, yr, yl;
  unsigned x0, x1, y0, y1;  // the box, in tiles (half open)
};

__device__ __forceinline__ Footprint footprint(const BinArgs &a, uint32_t g, uint2 rc) {
  Footprint f;
  const float4 m = a.smean[g], k = a.sconic[g];
  const float A = k.x, B = k.y, C = k.z;
  const float cut = (log2f(k.w / a.alpha_min) + 1e-3f) * 1.001f + 0.01f;
  const float D = fmaxf(4.f * A * C - B * B, 1e-30f);
  f.mx = m.x + m.z;
  f.my = m.y + m.w;
  f.bx = B / (2.f * A);         // x of the centre line: mx - bx dy
  f.cutA = cut / A;
  f.dA = D / (4.f * A * A);
  f.ry = sqrtf(cut * 4.f * A / D) * 1.0001f + 1e-3f;  // half extents
  f.rx = sqrtf(cut * 4.f * C / D) * 1.0001f + 1e-3f;
  const float by = B / (2.f * C);
  f.yr = f.my - by * f.rx;      // y of the rightmost point
  f.yl = f.my + by * f.rx;      // y of the leftmost point
  f.x0 = rc.x & 0xffffu;
  f.x1 = rc.x >> 16;
  f.y0 = rc.y & 0xffffu;
  f.y1 = rc.y >> 16;
  return f;
}

// Tiles [*lo, *hi) of row ty that the ellipse reaches (within the box).
__device__ __forceinline__ void row_span(const Footprint &f, unsigned ty, unsigned *lo,
                                         unsigned *hi) {
  *lo = *hi = f.x0;
  const float ya = fmaxf((float)(ty * kTile) + 0.5f, f.my - f.ry);
  const float yb = fminf((float)(ty * kTile) + (kTile - 0.5f), f.my + f.ry);
  if (ya > yb) return;
  auto hw = [&](float y) {
    const float d = y - f.my;
    return sqrtf(fmaxf(f.cutA - f.dA * d * d, 0.f));
  };
  const float ca = f.mx - f.bx * (ya - f.my), cb = f.mx - f.bx * (yb - f.my);
  const float wa = hw(ya), wb = hw(yb);
  const float xr = (f.yr >= ya && f.yr <= yb) ? f.mx + f.rx : fmaxf(ca + wa, cb + wb);
  const float xl = (f.yl >= ya && f.yl <= yb) ? f.mx - f.rx : fminf(ca - wa, cb - wb);
  // tile tx covers pixel centres [16 tx + 0.5, 16 tx + 15.5]
  const float tl = ceilf((xl - 1e-3f - (kTile - 0.5f)) / kTile);
  const float th = floorf((xr + 1e-3f - 0.5f) / kTile) + 1.f;
  const float l = fmaxf(tl, (float)f.x0), h = fminf(th, (float)f.x1);
  if (h > l) {
    *lo = (unsigned)l;
    *hi = (unsigned)h;
  }
}

__device__ __forceinline__ unsigned tiles_hit(const BinArgs &a, uint32_t g, uint2 rc) {
  const Footprint f = footprint(a, g, rc);
  unsigned c = 0;
  for (unsigned ty = f.y0; ty < f.y1; ++ty) {
    unsigned lo, hi;
    row_span(f, ty, &lo, &hi);
    c += hi - lo;
  }
  return c;
}

// One Gaussian per thread (kBinBlock per block): the block's sum of tile counts.
__global__ void __launch_bounds__(kBinBlock) count_kernel(BinArgs a) {
  griddep_enter();
  const int64_t i = (int64_t)blockIdx.x * kBinBlock + threadIdx.x;
  unsigned long long s = 0;
  if (i < a.n && !a.ctrl->gave_up) {  // (then there is no order)
    const uint32_t g = a.order[i];
    const uint2 rc = a.rect[g];
    if (rect_tiles(rc)) s = tiles_hit(a, g, rc);
    a.tiles[i] = (uint32_t)s;
  }
  unsigned long long tot;
  block_exclusive_scan(s, &tot);
  if (threadIdx.x == 0) a.blocksum[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) blocksum_scan_kernel(BinArgs a, int nb) {
  griddep_enter();
  __shared__ unsigned long long wt[32];
  const int per = (nb + 1023) / 1024;
  const int b = threadIdx.x * per, e = min(b + per, nb);
  unsigned long long s = 0;
  for (int i = b; i < e; ++i) s += a.blocksum[i];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned long long x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wt[w] = x;
  __syncthreads();
  if (w == 0) {
    unsigned long long t = wt[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    wt[lane] = t;
  }
  __syncthreads();
  unsigned long long run = x - s + (w > 0 ? wt[w - 1] : 0ull);
  for (int i = b; i < e; ++i) {
    const unsigned long long v = a.blocksum[i];
    a.blocksum[i] = run;
    run += v;
  }
  if (threadIdx.x == 1023) {
    const unsigned long long total = wt[31];
    a.ctrl->n_pairs = total;
    if (total > a.pair_cap) set_status(a.ctrl, GDGS_ERR_CAPACITY);
  }
}

// The lane that holds element i, from the lanes' inclusive counts (31 beyond the last).
__device__ __forceinline__ int owner(unsigned incl, unsigned i) {
  int o = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1)
    if (__shfl_sync(0xffffffffu, incl, o + step - 1) <= i) o += step;
  return min(o, 31);
}

// The pairs of kBinBlock depth-ordered Gaussians at a time, a warp's 32 in three steps: a
// lane per Gaussian (its footprint, to shared memory), a lane per row of tiles (its span), a
// lane per pair, so that the stores are whole lines (a thread per Gaussian wrote 32 scattered
// words a store: 16.4M pairs 165 us and 62 us more for the digit counts, now 91 us). Also counts the pairs' digits for the sort and
// clears what its first pass publishes.
__global__ void __launch_bounds__(kBinBlock) emit_kernel(BinArgs a, int nb) {
  griddep_enter();
  if (a.ctrl->gave_up) return;  // no order
  __shared__ Footprint s_f[kBinBlock];
  __shared__ unsigned s_bins[4][256];
  const int tid = threadIdx.x, lane = tid & 31, w0 = tid & ~31;
  for (int t = tid; t < 4 * 256; t += kBinBlock) (&s_bins[0][0])[t] = 0u;
  const unsigned np = item_count(&a.ctrl->n_pairs, a.pair_cap);
  clear_state(a.state, (np + kPairTile - 1) / kPairTile, pair_digits(a.digit), blockIdx.x * kBinBlock + tid, gridDim.x * kBinBlock);
  const unsigned mask = (1u << a.digit) - 1u, full = 0xffffffffu;
  for (int block = blockIdx.x; block < nb; block += gridDim.x) {
    const int64_t i = (int64_t)block * kBinBlock + tid;
    uint32_t g = 0;
    unsigned cnt = 0u, rows = 0u;
    if (i < a.n) {
      g = a.order[i];
      cnt = a.tiles[i];  // as counted by count_kernel
    }
    if (cnt) {
      const Footprint f = footprint(a, g, a.rect[g]);
      s_f[tid] = f;
      rows = f.y1 - f.y0;
    }
    unsigned long long tot;  // (its barriers also order s_bins)
    const unsigned long long my = a.blocksum[block] + block_exclusive_scan(cnt, &tot);
    unsigned long long at = __shfl_sync(full, my, 0);  // where the warp's next pair goes
    unsigned re = rows;  // rows of the warp's Gaussians up to this one
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned y = __shfl_up_sync(full, re, o);
      if (lane >= o) re += y;
    }
    const unsigned nrows = __shfl_sync(full, re, 31);
    for (unsigned r0 = 0; r0 < nrows; r0 += 32) {
      const unsigned r = r0 + lane;
      const int o = owner(re, r);
      const unsigned before = __shfl_sync(full, re - rows, o);
      const uint32_t rg = __shfl_sync(full, g, o);
      unsigned len = 0, key0 = 0;
      if (r < nrows) {
        const Footprint &f = s_f[w0 + o];
        const unsigned ty = f.y0 + (r - before);
        unsigned lo, hi;
        row_span(f, ty, &lo, &hi);
        len = hi - lo;
        key0 = ty * (unsigned)a.tiles_x + lo;
      }
      unsigned le = len;
#pragma unroll
      for (int k = 1; k < 32; k <<= 1) {
        const unsigned y = __shfl_up_sync(full, le, k);
        if (lane >= k) le += y;
      }
      const unsigned npairs = __shfl_sync(full, le, 31);
      // digits above the first: a row of tiles has one or two of each
      const unsigned long long p0 = at + (le - len);
      const unsigned kept = p0 >= a.pair_cap ? 0u : (unsigned)min((unsigned long long)len, a.pair_cap - p0);
      for (int p = 1; p < a.passes; ++p) {
        const int shift = p * a.digit;
        for (unsigned k = key0, end = key0 + kept; k < end;) {
          const unsigned next = min(end, ((k >> shift) + 1u) << shift);
          atomicAdd(&s_bins[p][(k >> shift) & mask], next - k);
          k = next;
        }
      }
      for (unsigned j0 = 0; j0 < npairs; j0 += 32) {
        const unsigned j = j0 + lane;
        const int q = owner(le, j);
        const uint32_t key = __shfl_sync(full, key0 - (le - len), q) + j, val = __shfl_sync(full, rg, q);
        const unsigned long long pos = at + j;
        if (j < npairs && pos < a.pair_cap) {
          a.pkey[pos] = key;
          a.pval[pos] = val;
          atomicAdd(&s_bins[0][key & mask], 1u);
        }
      }
      at += npairs;
    }
  }
  __syncthreads();
  for (int t = tid; t < a.passes * 256; t += kBinBlock) {
    const unsigned c = (&s_bins[0][0])[t];
    if (c) atomicAdd(&a.bins[t], c);
  }
}

}  // namespace

namespace {

template <int THREADS, int ITEMS>
constexpr int sort_smem() {
  return 4 * (2 * THREADS * ITEMS + THREADS / 32 * 512);
}

template <int THREADS, int ITEMS, int BITS, int kKind>
cudaError_t launch_pass(const SortPass &a, unsigned tiles, cudaStream_t st) {
  constexpr int smem = sort_smem<THREADS, ITEMS>();
  const auto kern = sort_pass_kernel<THREADS, ITEMS, BITS, kKind>;
  static_assert(smem <= 40 * 1024, "with the static arrays within 48 KB");
  LaunchScope ls_("radix_pass", st);
  launch_k(kern, std::min<unsigned>(tiles, kSortGrid), THREADS, smem, st, a);
  return cudaGetLastError();
}

template <int kKind>
cudaError_t launch_pair_pass(const SortPass &a, int digit, unsigned tiles, cudaStream_t st) {
  switch (digit) {
    case 8: return launch_pass<kPairThreads, kPairItems, 8, kKind>(a, tiles, st);
    case 7: return launch_pass<kPairThreads, kPairItems, 7, kKind>(a, tiles, st);
    case 6: return launch_pass<kPairThreads, kPairItems, 6, kKind>(a, tiles, st);
    default: return launch_pass<kPairThreads, kPairItems, 5, kKind>(a, tiles, st);
  }
}

unsigned pair_tiles(unsigned cap) { return (unsigned)(((unsigned long long)cap + kPairTile - 1) / kPairTile); }

// The words of one of two successive passes over at most `tiles` tiles (nobody reads those of
// a single one: one set for all passes).
SortState sort_state(uint32_t *base, int which, unsigned tiles, int digits) {
  const size_t groups = (tiles + kGroup - 1) / kGroup;
  uint32_t *p = base + (tiles > 1 ? which : 0) * digits * (tiles + 2 * groups);
  return {p, p + digits * tiles, p + digits * (tiles + groups)};
}

}  // namespace

size_t sort_state_words(long long keys, int tile, int digits, int passes) {
  const size_t tiles = (size_t)((keys + tile - 1) / tile), groups = (tiles + kGroup - 1) / kGroup;
  return (tiles > 1 ? std::min(passes, 2) : 1) * digits * (tiles + 2 * groups);
}

cudaError_t sort_depth(const DepthSort &s, cudaStream_t st) {
  const unsigned tiles = (unsigned)((s.n + kDepthTile - 1) / kDepthTile);
  if (tiles == 0) return cudaSuccess;
  {
    LaunchScope ls_("radix_hist", st);
    launch_k(depth_hist_kernel, std::min<unsigned>((s.n + 4 * kHistThreads - 1) / (4 * kHistThreads), kHistGrid),
             kHistThreads, 0, st, s, sort_state(s.state, 0, tiles, kDepthDigits));
  }
  for (int p = 0; p < kSortPasses; ++p) {
    SortPass a{};
    a.keys_in = p ? s.key[p & 1] : s.key_lo;
    a.vals_in = s.val[p & 1];
    a.keys_next = s.key[0];
    a.keys_out = s.key[~p & 1];
    a.vals_out = s.val[~p & 1];
    a.cap = s.n;
    a.shift = p ? 8 * (p - 1) : 0;
    a.bins = s.scratch.bins + 256 * p;
    a.ticket = s.scratch.ticket + p;
    a.state = sort_state(s.state, p & 1, tiles, kDepthDigits);
    if (p + 1 < kSortPasses) a.state_next = sort_state(s.state, ~p & 1, tiles, kDepthDigits);
    a.ctrl = s.ctrl;
    const cudaError_t e = p ? launch_pass<kDepthThreads, kDepthItems, 8, kSortPlain>(a, tiles, st)
                            : launch_pass<kDepthThreads, kDepthItems, 8, kSortLow>(a, tiles, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t sort_pairs(const PairSort &s, cudaStream_t st) {
  const unsigned tiles = pair_tiles(s.cap);
  if (tiles == 0) return cudaSuccess;
  const int passes = pair_passes(s.T), digit = pair_digit(s.T);
  for (int p = 0; p < passes; ++p) {
    SortPass a{};
    a.keys_in = s.key[p & 1];
    a.vals_in = s.val[p & 1];
    a.keys_out = s.key[~p & 1];
    a.vals_out = s.val[~p & 1];
    a.n_dev = s.n_dev;
    a.cap = s.cap;
    a.shift = p * digit;
    a.bins = s.scratch.bins + 256 * p;
    a.ticket = s.scratch.ticket + p;
    a.state = sort_state(s.state, p & 1, tiles, pair_digits(digit));
    if (p + 1 < passes) a.state_next = sort_state(s.state, ~p & 1, tiles, pair_digits(digit));
    a.ctrl = s.ctrl;
    a.range = s.range;
    a.active = s.active;
    a.tile_mask = s.tile_mask;
    const cudaError_t e = p + 1 < passes ? launch_pair_pass<kSortPlain>(a, digit, tiles, st)
                                         : launch_pair_pass<kSortRanges>(a, digit, tiles, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_emit_pairs(const BinArgs &b, cudaStream_t st) {
  if (b.n == 0) return cudaSuccess;
  BinArgs a = b;
  a.state = sort_state(b.sort_state, 0, pair_tiles(b.pair_cap), pair_digits(pair_digit(b.T)));
  a.passes = pair_passes(b.T);
  a.digit = pair_digit(b.T);
  const int nb = (int)((a.n + kBinBlock - 1) / kBinBlock);
  { LaunchScope ls_("pair_count", st); launch_k(count_kernel, nb, kBinBlock, 0, st, a); }
  { LaunchScope ls_("pair_scan", st); launch_k(blocksum_scan_kernel, 1, 1024, 0, st, a, nb); }
  { LaunchScope ls_("pair_emit", st); launch_k(emit_kernel, std::min(nb, kEmitGrid), kBinBlock, 0, st, a, nb); }
  return cudaGetLastError();
}

}  // namespace gdgs
