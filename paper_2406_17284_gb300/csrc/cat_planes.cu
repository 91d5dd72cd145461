// Host side of the bit-plane box-sum kernels (cat_planes.cuh): the kernel for
// a storage and radius, and the split of a grid into strips.
#include <atomic>

#include "cat_planes.cuh"

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
  planes::Params p;
  p.in = g.in;
  p.out = g.out;
  p.pitch = g.pitch;
  p.H = (int32_t)g.H;
  p.W = (int32_t)g.W;
  p.frame = g.frame;
  p.seg = (int32_t)((g.W + 2 * g.frame + 31) / 32) + 1;
  p.last = (uint32_t)(g.rule.C - 1) * 0x11111111u;
  p.two = g.rule.C > 2 ? 0x11111111u : 0u;
  set_bound(p.bound[planes::kSurviveLo], g.rule.s_lo, k.planes);
  set_bound(p.bound[planes::kSurviveHi], (int64_t)g.rule.s_lo + g.rule.s_w + 1, k.planes);
  set_bound(p.bound[planes::kBirthLo], g.rule.b_lo, k.planes);
  set_bound(p.bound[planes::kBirthHi], (int64_t)g.rule.b_lo + g.rule.b_w + 1, k.planes);
  // as many strips as fill the GPU once
  int64_t strips = (int64_t)resident * planes::kOut / p.seg;
  if (strips < 1) strips = 1;
  int64_t rows = (g.H + strips - 1) / strips;
  rows = (rows + k.ahead - 1) / k.ahead * k.ahead;
  strips = (g.H + rows - 1) / rows;
  p.rows = (int32_t)rows;
  p.strips = (int32_t)strips;
  const int64_t warps = (strips * p.seg + planes::kOut - 1) / planes::kOut;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)warps);
  cfg.blockDim = dim3(32);
  cfg.dynamicSmemBytes = (size_t)k.smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k.fn, p);
}

}  // namespace cat
