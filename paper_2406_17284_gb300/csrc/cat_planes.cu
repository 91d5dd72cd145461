// Host side of the bit-plane box-sum kernels (cat_planes.cuh): the kernel for
// a storage and radius, and the split of a grid into strips.
#include <algorithm>
#include <atomic>

#include "cat_planes_tile.cuh"

namespace cat {
namespace {

// The kernel for a grid's storages, and which of them it is (kinds x radii).
constexpr int kKinds = 6;
planes::Kernel find(const PlanesGrid &g, int *kind) {
  const int r = g.rule.r;
  const bool from_u8 = g.storage_in == CAT_STORE_U8, to_u8 = g.storage_out == CAT_STORE_U8;
  *kind = from_u8 && to_u8 ? (g.rule.C > 2 ? 1 : 0) : from_u8 ? 2 : to_u8 ? 3 : g.storage_in == CAT_STORE_BIT1 ? 4 : 5;
  if (g.rule.nbhd != 0 || r < 1 || r > planes::kMaxR || g.rule.C > 16) return planes::Kernel{};
  if (*kind >= 2 && *kind <= 4 && g.rule.C != 2) return planes::Kernel{};
  switch (*kind) {
    case 0: return planes::kernel_u8(r);
    case 1: return planes::kernel_u8_ms(r);
    case 2: return planes::kernel_u8_to_bit1(r);
    case 3: return planes::kernel_bit1_to_u8(r);
    case 4: return planes::kernel_bit1(r);
    default: return planes::kernel_nib4(r);
  }
}

// Warps of a kernel that the current device holds at once (looked up once per
// device, kind and radius; the value is a property of the device, so threads
// that race write the same).
cudaError_t resident_warps(const planes::Kernel &k, int kind, int r, const PlanesGrid &g, int *warps) {
  static std::atomic<int> seen[16][kKinds][planes::kMaxR + 1];
  std::atomic<int> *slot = g.device >= 0 && g.device < 16 ? &seen[g.device][kind][r] : nullptr;
  if (slot && (*warps = slot->load(std::memory_order_relaxed)) > 0) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, k.smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k.fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, 32, k.smem);
  if (e != cudaSuccess) return e;
  *warps = per_sm * g.sms;
  if (slot) slot->store(*warps, std::memory_order_relaxed);
  return cudaSuccess;
}

// A bound K of the rule as the words of a carry chain (planes::at_least), K
// clamped to [0, 2^planes): no count reaches 2^planes - 1 (an odd square is 1
// mod 8), so K = 2^planes - 1 means never.
void set_bound(uint32_t *k, int64_t K, int planes) {
  const int64_t top = (int64_t(1) << planes) - 1;
  const uint32_t c = ~(uint32_t)(K < 0 ? 0 : K > top ? top : K);
  for (int i = 0; i < planes; ++i) k[i] = 0u - ((c >> i) & 1u);
}

planes::Params make_params(const PlanesGrid &g, int planes) {
  planes::Params p;
  p.in = g.in;
  p.out = g.out;
  p.pitch = g.pitch;
  p.H = (int32_t)g.H;
  p.W = (int32_t)g.W;
  p.frame = g.frame;
  p.seg = (int32_t)((g.W + 2 * g.frame + 31) / 32) + 1;
  p.rows = p.strips = 0;
  p.last = (uint32_t)(g.rule.C - 1) * 0x11111111u;
  p.two = g.rule.C > 2 ? 0x11111111u : 0u;
  set_bound(p.bound[planes::kSurviveLo], g.rule.s_lo, planes);
  set_bound(p.bound[planes::kSurviveHi], (int64_t)g.rule.s_lo + g.rule.s_w + 1, planes);
  set_bound(p.bound[planes::kBirthLo], g.rule.b_lo, planes);
  set_bound(p.bound[planes::kBirthHi], (int64_t)g.rule.b_lo + g.rule.b_w + 1, planes);
  return p;
}

// A launch that may start while the one before it drains (the kernels wait for
// its end before they touch the grid).
template <typename P>
cudaError_t launch(void (*fn)(P), const P &p, int64_t blocks, int threads, int smem, cudaStream_t s) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, p);
}

constexpr int kMaxSmem = 232448;

// Steps before the words that a tile's warps write need a stale cell: the left
// neighbour word loses r cells a step; the right one r, and r more because the
// sums of a word are formed from the next word's shifted copy.
int max_tile_steps(int r) { return std::max(1, 32 / r - 1); }

// Output rows per strip (a multiple of 8) so that one wave of blocks holds the
// grid; 0 where not even one strip fits.
int32_t one_wave_rows(const PlanesGrid &g) {
  const int64_t strips = (int64_t)g.sms * planes::kOut / ((g.W + 31) / 32 + 1);
  return strips < 1 ? 0 : (int32_t)std::min<int64_t>(((g.H + strips - 1) / strips + 7) / 8 * 8, 1 << 20);
}

int64_t tile_smem(const PlanesGrid &g, const TilePlan &t) {
  const planes::TileKernel k = planes::tile_kernel(g.rule.r);
  return (int64_t)k.row_bytes * (t.rows + 2 * t.steps * g.rule.r) + k.block_bytes;
}

}  // namespace

// Where the bit planes are the faster path (us per step on GB300 against the
// tensor-core kernel that the options would otherwise name):
//   one bit per cell      every radius: 32768^2, r = 2 / 16: 147 / 320 against
//                         the former bit-sliced kernel's 224 and tcgen05's 594
//   four bits per cell    every radius: 24576^2, C 16, r = 10: 297 against 435
//   uint8, C > 2          24576^2, r = 10 / 16: 356 / 418 against 398: r <= 15
//   uint8, two states     only where a launch's latency counts: 1024^2, r = 1:
//                         2.9 against 6.5; 4096^2, r = 4 / 9 / 16: 9.5 / 14.8 /
//                         18.4 against 11.6 / 14.8 / 14.8; 16384^2, r = 4:
//                         111 against 97
bool planes_preferred(const PlanesGrid &g) {
  int kind;
  if (!find(g, &kind).fn) return false;
  if (g.storage_in != CAT_STORE_U8) return true;
  if (g.rule.C > 2) return g.rule.r <= 15;
  return g.rule.r <= 9 && g.H * g.W <= (1 << 24);
}

cudaError_t planes_launch(const PlanesGrid &g, cudaStream_t s) {
  int kind, resident;
  const planes::Kernel k = find(g, &kind);
  if (!k.fn) return cudaErrorInvalidValue;
  cudaError_t e = resident_warps(k, kind, g.rule.r, g, &resident);
  if (e != cudaSuccess) return e;
  planes::Params p = make_params(g, k.planes);
  // as many strips as fill the GPU once
  int64_t strips = (int64_t)resident * planes::kOut / p.seg;
  if (strips < 1) strips = 1;
  int64_t rows = (g.H + strips - 1) / strips;
  rows = (rows + k.ahead - 1) / k.ahead * k.ahead;
  strips = (g.H + rows - 1) / rows;
  p.rows = (int32_t)rows;
  p.strips = (int32_t)strips;
  const int64_t warps = (strips * p.seg + planes::kOut - 1) / planes::kOut;
  return launch(k.fn, p, warps, 32, k.smem, s);
}

// One wave of blocks, the strips as short as that allows, and k so that a
// launch's cost and the rows beside a strip that k steps need balance (us per
// step, streaming -> tiles: 256^2 to 1024^2, r = 1 / 4 / 9 / 16: 2.0 / 2.4 /
// 3.7 / 5.7 -> 0.8 / 1.8 / 3.0 / 4.3; 2048^2: 2.2 / 3.2 / 5.3 / 8.9 -> 1.3 /
// 2.7 / 4.4 / 6.1; 4096^2: 5.4 / 7.5 / 10.5 / 12.8 -> 3.1 / 5.9 / 9.3 / 12.5).
// A single step pays only where the streaming kernel's first 2r rows weigh
// more than two barriers (r >= 8).
TilePlan planes_tile_plan(const PlanesGrid &g, int64_t n_left) {
  const TilePlan none{0, 0};
  const int r = g.rule.r;
  if (g.rule.nbhd != 0 || r > planes::kMaxR || g.rule.C != 2 || g.storage_in == CAT_STORE_NIB4 || g.frame || n_left < 1)
    return none;
  const int most = std::min({8, std::max(1, 20 / r), max_tile_steps(r)});
  const int64_t launches = (n_left + most - 1) / most;
  const int steps = (int)((n_left + launches - 1) / launches);
  if (steps == 1 && r < 8) return none;
  const TilePlan t{steps, one_wave_rows(g)};
  return t.rows > 0 && tile_smem(g, t) <= kMaxSmem ? t : none;
}

// k steps per launch as asked for, on any grid: several waves of strips where
// one does not hold it.
TilePlan planes_tile_fixed(const PlanesGrid &g, int steps) {
  const TilePlan t{steps, one_wave_rows(g)};
  return t.rows > 0 && t.rows <= 128 ? t : TilePlan{steps, 64};
}

cudaError_t planes_tile_launch(const PlanesGrid &g, const TilePlan &plan, cudaStream_t s) {
  const planes::TileKernel k = planes::tile_kernel(g.rule.r);
  planes::TileParams t;
  t.p = make_params(g, k.planes);
  t.steps = plan.steps;
  t.in_u8 = g.storage_in == CAT_STORE_U8;
  t.out_u8 = g.storage_out == CAT_STORE_U8;
  t.p.rows = plan.rows;
  t.p.strips = (int32_t)((g.H + plan.rows - 1) / plan.rows);
  const int64_t smem = tile_smem(g, plan);
  if (!k.fn || plan.steps > max_tile_steps(g.rule.r) || smem > kMaxSmem) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e == cudaSuccess)   // (as the streaming kernels ask for: launches of both follow each other)
    e = cudaFuncSetAttribute(k.fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e != cudaSuccess) return e;
  const int64_t blocks = ((int64_t)t.p.strips * t.p.seg + planes::kOut - 1) / planes::kOut;
  return launch(k.fn, t, blocks, 32 * planes::kTileWarps, (int)smem, s);
}

}  // namespace cat
