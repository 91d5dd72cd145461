// Host side of the bit-plane box-sum kernels (cat_planes.cuh): the kernel for
// a storage and radius, and the split of a grid into strips.
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "cat_planes_tile.cuh"

namespace cat {
namespace planes {

// A bound K of the rule as the words of a carry chain (at_least), K clamped to
// [0, 2^planes): no count reaches 2^planes - 1 (an odd square is 1 mod 8), so
// K = 2^planes - 1 means never.
static void set_bound(uint32_t *k, int64_t K, int planes) {
  const int64_t top = (int64_t(1) << planes) - 1;
  const uint32_t c = ~(uint32_t)(K < 0 ? 0 : K > top ? top : K);
  for (int i = 0; i < planes; ++i) k[i] = 0u - ((c >> i) & 1u);
}

void set_bounds(uint32_t (*bound)[kMaxS], const RuleDev &rule, int planes) {
  set_bound(bound[kSurviveLo], rule.s_lo, planes);
  set_bound(bound[kSurviveHi], (int64_t)rule.s_lo + rule.s_w + 1, planes);
  set_bound(bound[kBirthLo], rule.b_lo, planes);
  set_bound(bound[kBirthHi], (int64_t)rule.b_lo + rule.b_w + 1, planes);
}

}  // namespace planes

namespace {

constexpr int kMaxSmem = 232448;   // of one block

// The kernel for a grid's storages, and which of them it is (kinds x radii).
constexpr int kKinds = 6;
planes::Kernel find(const PlanesGrid &g, int *kind) {
  const int r = g.rule.r;
  const bool from_u8 = g.storage_in == CAT_STORE_U8, to_u8 = g.storage_out == CAT_STORE_U8;
  *kind = from_u8 && to_u8 ? (g.rule.C > 2 ? 1 : 0) : from_u8 ? 2 : to_u8 ? 3 : g.storage_in == CAT_STORE_BIT1 ? 4 : 5;
  if (g.rule.nbhd != 0 || r < 1 || r > planes::kMaxR || g.rule.C > 16 || g.pitch > (int64_t)UINT32_MAX)
    return planes::Kernel{};
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

// Warps of a kernel that an SM of the current device holds, and the shared
// memory per warp that makes it so.  All warps have equal work, so an SM that
// takes one more than the others, or a scheduler of its four, is waited for:
// the warps per SM are a multiple of four, and a warp asks for as much shared
// memory as lets just that many in (one bit, 16384^2, r = 10 / 11 / 14: 14, 13
// and 10 warps 79 / 86 / 84 us a step, 12, 12 and 8 warps 69 / 71 / 71).  Looked
// up once per device, kind and radius; the values are a property of the
// device, so threads that race write the same.
struct Resident {
  int warps, smem;
};
constexpr int kSmSmem = 233472, kBlockReserve = 1024;   // bytes per SM, taken by the system per block

cudaError_t resident_warps(const planes::Kernel &k, int kind, int r, const PlanesGrid &g, Resident *out) {
  static std::atomic<int> seen[16][kKinds][planes::kMaxR + 1];
  std::atomic<int> *slot = g.device >= 0 && g.device < 16 ? &seen[g.device][kind][r] : nullptr;
  int per_sm = slot ? slot->load(std::memory_order_relaxed) : 0;
  if (per_sm == 0) {
    cudaError_t e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k.fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, 32, k.smem);
    if (e != cudaSuccess) return e;
    if (per_sm > 4 && per_sm % 4) per_sm = -(per_sm / 4 * 4);   // negative: only by asking for more
    if (slot) slot->store(per_sm, std::memory_order_relaxed);
  }
  const int n = std::max(1, std::abs(per_sm));
  out->warps = n * g.sms;
  out->smem = per_sm < 0 ? std::max(k.smem, (kSmSmem / n - kBlockReserve) / 128 * 128) : k.smem;
  return cudaSuccess;
}

planes::Params make_params(const PlanesGrid &g, int planes) {
  planes::Params p;
  p.in = g.in;
  p.out = g.out;
  p.pitch = g.pitch;
  p.H = (int32_t)g.H;
  p.W = p.written = (int32_t)g.W;
  p.frame = g.frame;
  p.seg = (int32_t)((g.W + 2 * g.frame + 31) / 32) + 1;
  p.rows = p.strips = 0;
  p.last = (uint32_t)(g.rule.C - 1) * 0x11111111u;
  p.two = g.rule.C > 2 ? 0x11111111u : 0u;
  planes::set_bounds(p.bound, g.rule, planes);
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

int64_t words_of(const PlanesGrid &g) { return (g.W + 2 * g.frame + 31) / 32 + 1; }   // of a row, the zero word too

// A grid in units of 2^20 cells, as a warp of 30 words counts them: a narrow
// grid's zero word and half empty last word take their share (a grid of 1024
// columns or more is its own cells).
int64_t mega_cells(const PlanesGrid &g) {
  return (g.H * std::max(g.W, 30 * words_of(g)) + (1 << 20) - 1) >> 20;
}

// The words pad a row by 7% more than the tiles' columns do, or it fills three
// words and most of one tile.
bool padded(const PlanesGrid &g) {
  return 100 * 32 * words_of(g) > 107 * ((g.W + 127) / 128 * 128) || (g.W > 80 && g.W <= 96);
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
//   four bits per cell    every radius: 24576^2, C 16, r = 10: 269 against 435
//   uint8, C > 2          up to a radius that falls while the strips get too
//                         short for the 2r rows before them and rises again with
//                         the size: 1024^2, r = 12 / 13: 5.9 / 6.6 against 6.0;
//                         2048^2, r = 5 / 6: 7.4 / 8.0 against 7.5; 4096^2, r =
//                         7 / 8: 14.4 / 17.1 against 14.8 / 15.3; 8192^2, r = 9
//                         / 10: 44.3 / 45.8 against 44.1; 16384^2, r = 1 / 10 /
//                         12 / 15: 117 / 154 / 157 / 172 against 153 / 159 ..
//   uint8, two states     only where a launch's latency counts: 1024^2, r = 1 /
//                         9 / 15: 2.2 / 3.7 / 4.3 against 4.5; 2048^2, r = 9 /
//                         10: 5.5 / 5.8 against 5.5; 4096^2, r = 4 / 5: 9.2 /
//                         10.3 against 9.9; 16384^2, r = 4: 111 against 92.
//                         The frame that a torus refreshes first costs a short
//                         step more: 1024^2, r = 7 / 9: 5.5 / 5.8 against 5.7;
//                         2048^2, r = 4 / 6: 6.4 / 7.5 against 7.1
// Narrow grids: where the words pad a row more than the tiles do, the tiles keep
// what they do faster (C = 16: 1048576 x 100, r = 4 / 9: 101 / 113 against 81 / 83;
// 932067 x 225, r = 9: 170 against 145; torus 1638400 x 128, r = 2 / 5: 258 / 268
// against 202; two states 37282 x 225, r = 4: 10.7 against 8.9).  Up to 64 columns it is the other way round, three words
// against a tile of which half is outside the grid (C = 16: 1092266 x 48, r = 10 /
// 16: 63 / 75 against 109; 32768 x 48, r = 16: 12.6 against 9.6).
bool planes_preferred(const PlanesGrid &g) {
  int kind;
  if (!find(g, &kind).fn) return false;
  if (g.storage_in != CAT_STORE_U8) return true;
  const int64_t m = mega_cells(g);
  const bool narrow = padded(g), odd = g.W % 16 != 0;
  const int r = g.rule.r;
  if (g.rule.C > 2) {
    if (!g.frame && g.W <= 64 && m >= 24) return true;
    if (narrow && m >= 16)
      return r <= (g.frame ? (m < 64 ? (g.W <= 128 ? 3 : 5) : g.W <= 256 ? 0 : 5) : m < 64 ? 5 : g.W <= 128 && odd ? 0 : 7);
    return r <= (m <= 1 ? (g.frame ? 9 : 12) : m < 16 ? 5 : m < 64 ? 7 : m < 128 ? 9 : 12);
  }
  if (g.frame) return r <= (m <= 1 ? 7 : m <= 16 ? (narrow ? 2 : 4) : 0);
  return r <= (m <= 1 ? 16 : m <= 4 ? 9 : m <= 16 ? (narrow && odd ? 2 : 4) : 0);
}

// Several steps of a two-state uint8 grid (us per step, tensor-core steps
// last).  Reading and writing bits is worth most on large grids and with many
// steps between the bytes at both ends; a wave of strips fits grids of 6 to 50
// 2^20 cells badly, and a torus pays for a frame per launch:
//   2896^2, n = 2 / 4 / 8   r = 10: 8.1 / 6.8 / 6.7 and 7.9; r = 12: 8.2 / 8.0 /
//                           7.8 and 7.9
//   4096^2, n = 2 / 4 / 8   r = 4: 9.4 / 7.3 / 5.8 and 9.9; r = 7: 11.2 / 7.7 /
//                           7.5 and 9.9; r = 10: 11.7 / 9.5 / 9.3 and 9.9;
//                           r = 12: 12.0 / 11.5 / 11.3 and 9.9
//   5792^2, n = 2 / 4 / 8   r = 8: 18.5 / 16.3 / 15.3 and 16.7; r = 16: 22.0 /
//                           19.9 / 18.7 and 19.0
//   7000^2, n = 2 / 3 / 4   r = 12: 24.0 / 22.5 / 21.7 and 22.8; r = 16: 27.8 /
//                           25.8 / 24.6 and 24.8
//   8192^2, n = 2 / 3 / 8   r = 4: 20.1 / 18.8 / 17.3 and 27.2; r = 8: 29.2 / 27.0
//                           / 24.0 and 28.2; r = 16: 33.5 / 31.3 / 28.3 and 32.1
//   16384^2, n = 2 / 8      r = 12: 92.6 / 75.5 and 98.5
//   narrow, n = 2 / 3 / 8   1048576 x 100, r = 4: 75.8 / 71.2 / 53.0 and 60.0;
//                           1638400 x 128, r = 7: 105 / 106 / 95 and 73; 873813 x
//                           96, r = 3: 48.0 / 47.5 / .. and 41.8 (n = 5: 40.7); 362539
//                           x 376, r = 16: .. / 69.2 / .. and 59.9; torus 65536 x
//                           96, r = 7: .. / 15.3 / 16.1 and 12.3; torus 384362 x
//                           320, r = 13: 99 / .. / .. and 90
//   torus, n = 8            2048^2, r = 12: 9.0 and 7.1; 4096^2, r = 7 / 12: 10.9
//                           / 14.6 and 12.1; 5792^2, r = 12: 18.0 and 18.7;
//                           7000^2, r = 11 / 15: 23.6 / 22.7 and 23.4
bool planes_steps_preferred(const PlanesGrid &g, int64_t n_steps) {
  const int64_t m = mega_cells(g);
  const bool odd = g.W % 16 != 0;
  const int r = g.rule.r;
  if (padded(g) && g.frame) {
    if (m > 4 && m <= 36 && r > 4) return false;
    if (m > 12 && g.W <= 128) return false;
    if (m > 36) return r <= 4 || n_steps >= 8;
  } else if (padded(g) && m > 24) {
    if (g.W <= 96) return n_steps >= (m > 64 && odd ? 8 : 4);
    return n_steps >= 8 && (g.W > 128 || (r <= 4 && m <= 64));
  }
  if (g.frame) return r <= 7 || (m >= 30 && n_steps >= (m < 64 ? 8 : r == 8 || r >= (g.W < 512 ? 10 : 14) ? 3 : 2));
  if (r <= 7) return m <= 4 || m > 24 || n_steps >= (r == 7 ? 4 : r >= 5 ? 3 : 2);
  if (m <= (r <= 10 ? 10 : 6)) return true;
  if (m <= 24) return r <= 10 && n_steps >= 4;
  if (m <= 36) return n_steps >= (r == 16 ? 8 : 4);
  return n_steps >= (m <= 50 || r == 8 || r == 16 ? 3 : 2);
}

namespace {

// The tile kernel's shared memory and carveout (the latter as the streaming
// kernels ask for: launches of both follow each other), once per device.
cudaError_t tile_attributes(const planes::TileKernel &k, const PlanesGrid &g) {
  static std::atomic<bool> set[16][planes::kMaxR + 1];
  std::atomic<bool> *slot = g.device >= 0 && g.device < 16 ? &set[g.device][g.rule.r] : nullptr;
  if (slot && slot->load(std::memory_order_relaxed)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k.fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess && slot) slot->store(true, std::memory_order_relaxed);
  return e;
}

}  // namespace

cudaError_t planes_prepare(const PlanesGrid &g, const TilePlan &plan) {
  if (plan.steps > 0) {
    const planes::TileKernel k = planes::tile_kernel(g.rule.r);
    if (!k.fn || plan.steps > max_tile_steps(g.rule.r) || tile_smem(g, plan) > kMaxSmem || g.pitch > (int64_t)UINT32_MAX)
      return cudaErrorInvalidValue;
    return tile_attributes(k, g);
  }
  int kind;
  Resident resident;
  const planes::Kernel k = find(g, &kind);
  return k.fn ? resident_warps(k, kind, g.rule.r, g, &resident) : cudaErrorInvalidValue;
}

// A one-bit grid of a row or a few, too wide for one wave of warps: a warp here
// sums 2r rows and steps four (or eight) for those it writes, and a word to a
// thread with the rows in registers is the faster way (us a step, this / that: 1 x
// 2^20, r = 2: 3.2 / 2.0; 1 x 100 * 2^20, r = 1 / 2 / 5: 111 / 29, 111 / 46, 190 /
// 167; 5 x 100 * 2^20, r = 2 / 3: 157 / 136, 166 / 192; 2 x 100 * 2^20, r = 3 / 5: 111 /
// 108, 191 / 217).
bool planes_few_rows(const PlanesGrid &g) {
  return g.storage_in == CAT_STORE_BIT1 && g.W >= 1 << 19 && g.H <= 5 && g.rule.r <= (g.H == 1 ? 5 : g.H == 2 ? 4 : 2);
}

cudaError_t planes_launch(const PlanesGrid &g, cudaStream_t s) {
  int kind;
  Resident resident;
  const planes::Kernel k = find(g, &kind);
  if (!k.fn) return cudaErrorInvalidValue;
  cudaError_t e = resident_warps(k, kind, g.rule.r, g, &resident);
  if (e != cudaSuccess) return e;
  planes::Params p = make_params(g, k.planes);
  // as many strips as fill the GPU once
  int64_t strips = (int64_t)resident.warps * planes::kOut / p.seg;
  if (strips < 1) strips = 1;
  int64_t rows = (g.H + strips - 1) / strips;
  rows = (rows + k.ahead - 1) / k.ahead * k.ahead;
  strips = (g.H + rows - 1) / rows;
  p.rows = (int32_t)rows;
  p.strips = (int32_t)strips;
  const int64_t warps = (strips * p.seg + planes::kOut - 1) / planes::kOut;
  return launch(k.fn, p, warps, 32, resident.smem, s);
}

// One wave of blocks, the strips as short as that allows, and k so that a
// launch's cost and the rows beside a strip that k steps need balance (us per
// step, streaming -> tiles: 256^2 to 1024^2, r = 1 / 4 / 9 / 16: 2.0 / 2.4 /
// 3.7 / 5.7 -> 0.8 / 1.8 / 3.0 / 4.3; 2048^2: 2.2 / 3.2 / 5.3 / 8.9 -> 1.3 /
// 2.7 / 4.4 / 6.1; 4096^2: 5.4 / 7.5 / 10.5 / 12.8 -> 3.1 / 5.9 / 9.3 / 12.5).
// A single step pays only where the streaming kernel's first 2r rows weigh
// more than two barriers (r >= 8).
static int64_t fewest_launches(int r, int64_t n_steps) {
  const int most = std::min({8, std::max(1, 20 / r), max_tile_steps(r)});
  return (n_steps + most - 1) / most;
}

TilePlan planes_tile_steps(const PlanesGrid &g, int64_t steps) {
  const TilePlan none{0, 0};
  const int r = g.rule.r;
  if (g.rule.nbhd != 0 || r > planes::kMaxR || g.rule.C != 2 || g.storage_in == CAT_STORE_NIB4 || g.frame || steps < 1 ||
      steps > max_tile_steps(r))
    return none;
  if (steps == 1 && r < 8) return none;
  const TilePlan t{(int32_t)steps, one_wave_rows(g)};
  return t.rows > 0 && tile_smem(g, t) <= kMaxSmem ? t : none;
}

TilePlan planes_tile_plan(const PlanesGrid &g, int64_t n_left) {
  if (n_left < 1 || g.rule.r > planes::kMaxR) return TilePlan{0, 0};
  const int64_t launches = fewest_launches(g.rule.r, n_left);
  return planes_tile_steps(g, (n_left + launches - 1) / launches);
}

int64_t planes_launches(const PlanesGrid &g, int64_t n_steps) {
  int64_t launches = fewest_launches(g.rule.r, n_steps);
  launches += (launches ^ n_steps) & 1;   // (at most n_steps)
  return planes_tile_steps(g, (n_steps + launches - 1) / launches).steps > 0 ? launches : n_steps;
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
  const cudaError_t e = planes_prepare(g, plan);
  if (e != cudaSuccess) return e;
  const int64_t blocks = ((int64_t)t.p.strips * t.p.seg + planes::kOut - 1) / planes::kOut;
  return launch(k.fn, t, blocks, 32 * planes::kTileWarps, (int)tile_smem(g, plan), s);
}

struct PlanesBatch {
  struct Chain {
    int range;                            // of radii (planes::kRangeEnd)
    int smem;                             // of the largest radius
    unsigned blocks;                      // blocks of one launch (planes::kBatchWarps warps each)
    const planes::BatchBlock *first;
  };
  std::vector<Chain> chains;
  unsigned pack_blocks = 0;               // blocks that pack or unpack all grids
  const planes::BatchBlock *pack_first = nullptr;
  std::vector<planes::BatchGrid> grids;
  planes::BatchGrid *d_grids = nullptr;   // the lists of blocks follow in the same allocation
};

namespace {

// Rows per strip of a batch: about this many warps per SM over all grids, so
// that the 2r rows before a strip's first output row stay a small part (512
// uneven grids: 32 / 48 / 64 / 96 rows: 467 / 465 / 466 / 518 us).
constexpr int kBatchFill = 24;

planes::BatchParams batch_params(const PlanesBatch *b, const planes::BatchBlock *first, int64_t step, int64_t steps,
                                 int flip) {
  return planes::BatchParams{b->d_grids, first, flip, (int32_t)step, (int32_t)steps};
}

}  // namespace

static void set_buffers(PlanesBatch *b, const std::vector<PlanesBatchItem> &items) {
  for (size_t i = 0; i < items.size(); ++i) {
    b->grids[i].buf[0] = items[i].buf[0];
    b->grids[i].buf[1] = items[i].buf[1];
    b->grids[i].cur = items[i].cur;
  }
}

cudaError_t planes_batch_update(PlanesBatch *b, const std::vector<PlanesBatchItem> &items) {
  set_buffers(b, items);
  return cudaMemcpy(b->d_grids, b->grids.data(), sizeof(planes::BatchGrid) * b->grids.size(), cudaMemcpyHostToDevice);
}

cudaError_t planes_batch_create(const std::vector<PlanesBatchItem> &items, int sms, PlanesBatch **out) {
  PlanesBatch *b = new (std::nothrow) PlanesBatch();
  if (!b) return cudaErrorMemoryAllocation;
  double warp_rows = 0;
  for (const PlanesBatchItem &q : items) warp_rows += (double)q.H * ((q.W + 31) / 32 + 1) / planes::kOut;
  const int64_t rows = std::max<int64_t>(32, std::min<int64_t>(512, (int64_t)(warp_rows / (kBatchFill * sms)) / 4 * 4));
  b->grids.resize(items.size());
  std::vector<int32_t> of_radius[planes::kMaxR + 1];
  for (size_t i = 0; i < items.size(); ++i) {
    const PlanesBatchItem &q = items[i];
    planes::BatchGrid &g = b->grids[i];
    g = planes::BatchGrid{};
    g.pitch = q.pitch;
    g.H = (int32_t)q.H;
    g.W = (int32_t)q.W;
    g.seg = (int32_t)((q.W + 31) / 32) + 1;
    g.rows = (int32_t)std::min<int64_t>(rows, (q.H + 3) / 4 * 4);
    g.strips = (int32_t)((q.H + g.rows - 1) / g.rows);
    g.second = q.second;
    g.r = q.rule.r;
    of_radius[g.r].push_back((int32_t)i);
    planes::set_bounds(g.bound, q.rule, planes::kernel_bit1(q.rule.r).planes);
  }
  std::vector<planes::BatchBlock> blocks;
  std::vector<size_t> first;
  size_t most = planes::kMaxR * planes::kBatchWarps;
  for (const planes::BatchGrid &g : b->grids)
    most += (size_t)((int64_t)g.strips * g.seg / planes::kOut + (int64_t)g.H * g.seg / planes::kPackWords + 2);
  blocks.reserve(most);
  for (int r = planes::kMaxR; r >= 1; --r) {   // (the larger radii, whose blocks take longest, first)
    int range = 0;
    while (r > planes::kRangeEnd[range]) ++range;
    const size_t at = blocks.size();
    for (const int32_t i : of_radius[r]) {
      const int64_t n = ((int64_t)b->grids[i].strips * b->grids[i].seg + planes::kOut - 1) / planes::kOut;
      for (int64_t k = 0; k < n; ++k) blocks.push_back(planes::BatchBlock{i, (int32_t)k});
    }
    if (blocks.size() == at) continue;
    while (blocks.size() % planes::kBatchWarps) blocks.push_back(planes::BatchBlock{-1, 0});
    if (b->chains.empty() || b->chains.back().range != range) {
      b->chains.push_back(PlanesBatch::Chain{range, planes::kBatchWarps * planes::kernel_bit1(r).smem, 0u, nullptr});
      first.push_back(at);
    }
    b->chains.back().blocks += (unsigned)((blocks.size() - at) / planes::kBatchWarps);
  }
  const size_t pack_at = blocks.size();
  for (size_t i = 0; i < items.size(); ++i) {
    const int64_t words = (int64_t)b->grids[i].H * (b->grids[i].seg - 1);
    for (int64_t k = 0; k * planes::kPackWords < words; ++k) blocks.push_back(planes::BatchBlock{(int32_t)i, (int32_t)k});
  }
  b->pack_blocks = (unsigned)(blocks.size() - pack_at);
  const size_t grid_bytes = (sizeof(planes::BatchGrid) * b->grids.size() + 255) / 256 * 256;
  const size_t block_bytes = sizeof(planes::BatchBlock) * blocks.size();
  cudaError_t e = blocks.size() > 0x7fffffffu ? cudaErrorInvalidValue
                                              : cudaMalloc(&b->d_grids, grid_bytes + block_bytes);
  planes::BatchBlock *d_blocks =
      reinterpret_cast<planes::BatchBlock *>(reinterpret_cast<uint8_t *>(b->d_grids) + grid_bytes);
  if (e == cudaSuccess) {   // (one copy: each waits for the device)
    set_buffers(b, items);
    std::vector<uint8_t> table(grid_bytes + block_bytes);
    memcpy(table.data(), b->grids.data(), sizeof(planes::BatchGrid) * b->grids.size());
    memcpy(table.data() + grid_bytes, blocks.data(), block_bytes);
    e = cudaMemcpy(b->d_grids, table.data(), table.size(), cudaMemcpyHostToDevice);
  }
  b->pack_first = d_blocks + pack_at;
  for (size_t c = 0; c < b->chains.size() && e == cudaSuccess; ++c) {
    b->chains[c].first = d_blocks + first[c];
    const planes::BatchFn fn = planes::batch_kernel(b->chains[c].range);
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  }
  if (e != cudaSuccess) {
    planes_batch_free(b);
    return e;
  }
  *out = b;
  return cudaSuccess;
}

void planes_batch_free(PlanesBatch *b) {
  if (!b) return;
  cudaFree(b->d_grids);
  delete b;
}

cudaError_t planes_batch_add(const PlanesBatch *b, int64_t n_steps, int flip, cudaGraph_t graph) {
  const auto add = [&](planes::BatchFn fn, planes::BatchParams p, unsigned blocks, int threads, int smem,
                       const std::vector<cudaGraphNode_t> &after, cudaGraphNode_t *node) {
    void *args[1] = {&p};
    cudaKernelNodeParams k = {};
    k.func = reinterpret_cast<void *>(fn);
    k.gridDim = dim3(blocks);
    k.blockDim = dim3((unsigned)threads);
    k.sharedMemBytes = (unsigned)smem;
    k.kernelParams = args;
    return cudaGraphAddKernelNode(node, graph, after.data(), after.size(), &k);
  };
  cudaGraphNode_t pack{}, unpack{};
  cudaError_t e = add(planes::batch_pack_kernel(false), batch_params(b, b->pack_first, 0, n_steps, flip), b->pack_blocks,
                      planes::kPackThreads, 0, {}, &pack);
  std::vector<cudaGraphNode_t> ends;
  for (const PlanesBatch::Chain &c : b->chains) {   // the ranges of radii side by side
    cudaGraphNode_t before = pack;
    for (int64_t t = 0; t < n_steps && e == cudaSuccess; ++t)
      e = add(planes::batch_kernel(c.range), batch_params(b, c.first, t, n_steps, flip), c.blocks,
              32 * planes::kBatchWarps, c.smem, {before}, &before);
    ends.push_back(before);
  }
  if (e == cudaSuccess)
    e = add(planes::batch_pack_kernel(true), batch_params(b, b->pack_first, n_steps, n_steps, flip), b->pack_blocks,
            planes::kPackThreads, 0, ends, &unpack);
  return e;
}

}  // namespace cat
