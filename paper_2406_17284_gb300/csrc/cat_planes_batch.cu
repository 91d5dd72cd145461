// Batches on bit planes (cat_planes.cuh): the step kernels, and packing the
// states of all grids to bits and back.
#include "cat_planes.cuh"

namespace cat {
namespace planes {
namespace {

// A thread takes 32-cell words of one grid, a warp 32 consecutive ones (1 KiB
// of bytes); bound by the bytes (512 uneven grids, 161 MB: see batch_step).
template <bool UNPACK>
__global__ void __launch_bounds__(kPackThreads) batch_pack(const __grid_constant__ BatchParams b) {
  const int2 at = __ldg(reinterpret_cast<const int2 *>(b.blocks) + blockIdx.x);
  const BatchGrid *g = b.grids + at.x;
  const int cur = __ldg(&g->cur) ^ b.flip, H = __ldg(&g->H), W = __ldg(&g->W), words = __ldg(&g->seg) - 1;
  const int64_t pitch = __ldg(reinterpret_cast<const long long *>(&g->pitch));
  uint8_t *const bits = packed_place(g, cur, b.step, b.steps);
  uint8_t *const cells = reinterpret_cast<uint8_t *>(
      __ldg(reinterpret_cast<const unsigned long long *>(&g->buf[UNPACK ? cur ^ (b.steps & 1) : cur])));
  const int64_t first = (int64_t)at.y * kPackWords;
  const int row = (int)(first / words);
  const uint32_t skip = (uint32_t)(first - (int64_t)row * words);   // (one wide division per block)
#pragma unroll 4
  for (int k = 0; k < kPackWords; k += kPackThreads) {
    const uint32_t i = skip + (uint32_t)k + threadIdx.x, down = i / (uint32_t)words;
    const int y = row + (int)down, w = (int)(i - down * (uint32_t)words), left = W - 32 * w;
    if (y >= H) continue;
    uint8_t *const q = cells + y * pitch + 32 * w;
    uint32_t *const p = reinterpret_cast<uint32_t *>(bits + y * pitch) + w;
    if (UNPACK) {
      uint32_t o[4];
      const uint32_t f = *p, lo = f & 0x0F0F0F0Fu, hi = (f >> 4) & 0x0F0F0F0Fu;
      spread_bytes<0>(lo, hi, o);
      *reinterpret_cast<uint4 *>(q) = make_uint4(o[0], o[1], o[2], o[3]);
      spread_bytes<1>(lo, hi, o);
      if (left > 16) *reinterpret_cast<uint4 *>(q + 16) = make_uint4(o[0], o[1], o[2], o[3]);
    } else {
      Raw<CAT_STORE_U8> r;
      ld16(r.v, q);
      ld16(r.v + 4, left > 16 ? q + 16 : q);
      if (left < 32) {   // bytes past W are not the grid's
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c = left - 4 * j;
          r.v[j] &= c >= 4 ? ~0u : c <= 0 ? 0u : (1u << (8 * c)) - 1u;
        }
      }
      *p = flags<CAT_STORE_U8, false>(r);
    }
  }
}

}  // namespace

BatchFn batch_kernel(int range) {
  return range == 0   ? planes_batch_kernel<1, kRangeEnd[0]>
         : range == 1 ? planes_batch_kernel<kRangeEnd[0] + 1, kRangeEnd[1]>
                      : planes_batch_kernel<kRangeEnd[1] + 1, kRangeEnd[2]>;
}
BatchFn batch_pack_kernel(bool unpack) { return unpack ? batch_pack<true> : batch_pack<false>; }

}  // namespace planes
}  // namespace cat
