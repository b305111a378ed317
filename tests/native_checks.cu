// Checks of device code that the C interface does not reach, compiled by test_gpu_native.py
// together with the library's sources: `sort` the sorts behind a wait that gave up, `div` the
// backward rasteriser's packed division. Prints "ok" or what is wrong.
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "../paper_2405_05446_gb300/csrc/backward.cu"
#include "../paper_2405_05446_gb300/csrc/sort.cu"

using namespace gdgs;

namespace gdgs {
unsigned long long graph_kernel_count() { return 0; }  // (diag.cu asks the solver for it)
}

template <class T>
struct Buf {
  T *p = nullptr;
  size_t n;
  explicit Buf(size_t count, int byte = 0) : n(count) {
    if (cudaMalloc(&p, n * sizeof(T)) == cudaSuccess) cudaMemset(p, byte, n * sizeof(T));
  }
  void put(const std::vector<T> &v) { cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice); }
  std::vector<T> get() const {
    std::vector<T> v(n);
    cudaMemcpy(v.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost);
    return v;
  }
};

// The binning of n splats over 64 x 32 tiles, each reaching about 2 x 2 of them; with `gave_up`
// behind a status that already holds another error. Every index left in the buffers is 1.
static int run_sort(bool gave_up) {
  const unsigned n = 6000, tx = 64, T = 64 * 32, cap = 16 * n;
  std::vector<float4> mean(n), conic(n);
  std::vector<uint2> rect(n);
  std::vector<uint32_t> key(n), lo(n), ones_n(n, 1u), ones_c(cap, 1u);
  unsigned seed = 12345;
  auto rnd = [&] { return (seed = seed * 1664525u + 1013904223u) >> 8; };
  for (unsigned i = 0; i < n; ++i) {
    const unsigned cx = 1 + rnd() % 62, cy = 1 + rnd() % 30;
    mean[i] = make_float4(16.f * cx, 16.f * cy, 0.f, 0.f);  // a tile corner
    conic[i] = make_float4(0.05f, 0.f, 0.05f, 0.9f);
    rect[i] = make_uint2((cx - 1) | (cx + 1) << 16, (cy - 1) | (cy + 1) << 16);
    key[i] = 0x3f800000u + rnd() % 3000;
    lo[i] = rnd() & 255u;
  }
  Buf<float4> d_mean(n), d_conic(n);
  Buf<uint2> d_rect(n), range(T, 0xff);
  Buf<uint32_t> k0(n), k1(n), v0(n), v1(n), d_lo(n), pk0(cap), pk1(cap), pv0(cap), pv1(cap), tiles(n), active(T);
  Buf<uint32_t> state(std::max(sort_state_words(n, kDepthTile, kDepthDigits, kSortPasses),
                               sort_state_words(cap, kPairTile, pair_digits(pair_digit(T)), pair_passes(T))));
  Buf<uint32_t> scratch(sort_words(T));
  Buf<uint8_t> mask(T, 0xff);
  Buf<unsigned long long> blocksum((n + kBinBlock - 1) / kBinBlock + 2);
  Buf<Ctrl> ctrl(1);
  d_mean.put(mean), d_conic.put(conic), d_rect.put(rect), k0.put(key), d_lo.put(lo);
  for (auto *b : {&k1, &v0, &v1, &tiles}) b->put(ones_n);
  for (auto *b : {&pk0, &pk1, &pv0, &pv1}) b->put(ones_c);
  Ctrl c;
  memset(&c, 0, sizeof(c));
  if (gave_up) {
    c.status = GDGS_ERR_CAPACITY;
    c.gave_up = 1;
  }
  ctrl.put({c});
  DepthSort ds{};
  ds.key[0] = k0.p, ds.key[1] = k1.p, ds.val[0] = v0.p, ds.val[1] = v1.p;
  ds.key_lo = d_lo.p;
  ds.n = n;
  ds.state = state.p;
  ds.scratch = depth_scratch(scratch.p);
  ds.range = range.p, ds.tile_mask = mask.p, ds.T = T, ds.ctrl = ctrl.p;
  BinArgs b{};
  b.order = v1.p, b.rect = d_rect.p, b.smean = d_mean.p, b.sconic = d_conic.p;
  b.alpha_min = 1.f / 255.f, b.n = n, b.tiles_x = tx, b.T = T, b.pair_cap = cap;
  b.blocksum = blocksum.p, b.tiles = tiles.p, b.pkey = pk0.p, b.pval = pv0.p;
  b.bins = pair_scratch(scratch.p).bins, b.sort_state = state.p, b.ctrl = ctrl.p;
  PairSort ps{};
  ps.key[0] = pk0.p, ps.key[1] = pk1.p, ps.val[0] = pv0.p, ps.val[1] = pv1.p;
  ps.n_dev = (const unsigned long long *)((char *)ctrl.p + offsetof(Ctrl, n_pairs));
  ps.cap = cap, ps.T = T, ps.state = state.p;
  ps.scratch = pair_scratch(scratch.p);
  ps.range = range.p, ps.active = active.p, ps.tile_mask = mask.p, ps.ctrl = ctrl.p;
  if (sort_depth(ds, 0) != cudaSuccess || launch_emit_pairs(b, 0) != cudaSuccess || sort_pairs(ps, 0) != cudaSuccess ||
      cudaDeviceSynchronize() != cudaSuccess) {
    printf("launch: %s\n", cudaGetErrorString(cudaGetLastError()));
    return 1;
  }
  c = ctrl.get()[0];
  const auto order = v1.get(), pk = pk0.get(), pv = pv0.get(), sc = scratch.get();
  const auto rg = range.get();
  if (gave_up) {
    bool same = c.n_pairs == 0 && c.n_active == 0 && c.status == GDGS_ERR_CAPACITY && order == ones_n && pk == ones_c && pv == ones_c;
    for (int i = 0; i < 16; ++i) same = same && sc[kSortPasses * 256 + i] == 0u;  // the tickets
    for (const uint2 &r : rg) same = same && r.x == 0u && r.y == 0u;
    if (!same) printf("a pass ran behind a wait that gave up\n");
    return same ? 0 : 1;
  }
  // what the harness itself feeds is sorted: every tile's list by (key, lo, index)
  auto before = [&](uint32_t x, uint32_t y) { return key[x] != key[y] ? key[x] < key[y] : lo[x] != lo[y] ? lo[x] < lo[y] : x < y; };
  unsigned long long total = 0;
  for (unsigned t = 0; t < T; ++t) {
    if (!rg[t].y) continue;
    const unsigned s = ~rg[t].x, e = rg[t].y;
    total += e - s;
    for (unsigned i = s + 1; i < e; ++i)
      if (!before(pv[i - 1], pv[i])) return printf("tile %u is not in order\n", t), 1;
  }
  if (c.status != GDGS_OK || total != c.n_pairs || total != 4ull * n) return printf("%llu of %llu pairs\n", total, c.n_pairs), 1;
  return 0;
}

__global__ void div_kernel(unsigned long long *bad, int exponents, float lo) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long wrong = 0, x = t * 0x9e3779b97f4a7c15ull + 1;
  for (int i = 0; i < 1024; ++i) {
    x = x * 6364136223846793005ull + 1442695040888963407ull;
    const unsigned u = (unsigned)(x >> 32);
    x = x * 6364136223846793005ull + 1442695040888963407ull;
    const unsigned v = (unsigned)(x >> 32);
    const float a = ldexpf(1.f + (u >> 9) * 0x1p-23f, -1 - (int)(u % exponents));
    const float b = fmaxf(lo, lo + (1.f - lo) * (v >> 8) * 0x1p-24f);
    float q0, q1;
    unpk(div2(pk(a, a), pk(b, 1.f)), q0, q1);
    wrong += q0 != __fdiv_rn(a, b) || q1 != a;
  }
  if (wrong) atomicAdd(bad, wrong);
}

int main(int argc, char **argv) {
  int bad = 0;
  if (argc > 1 && !strcmp(argv[1], "sort")) bad = run_sort(false) || run_sort(true);
  if (argc > 1 && !strcmp(argv[1], "div")) {
    // transmittances of 1 .. 2^-100 over 1 - alpha for every alpha_max that the options take
    for (float lo : {0.01f, 1e-3f, 0x1p-24f}) {
      Buf<unsigned long long> n(1);
      div_kernel<<<304, 256>>>(n.p, 100, lo);
      const unsigned long long wrong = n.get()[0];
      if (cudaGetLastError() != cudaSuccess || wrong) printf("%llu quotients differ above %g\n", wrong, lo), bad = 1;
    }
  }
  if (!bad) printf("ok\n");
  return bad;
}
