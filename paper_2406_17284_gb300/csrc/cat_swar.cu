// Box counts of a one-bit grid by bit-sliced (SWAR) adders, radii 1..5: the
// verification path of the bit-sliced kernel choice, and its step on grids of a
// few very wide rows (the other steps run on cat_planes.cuh).
//
// Every 32-bit word of a packed row holds 32 cells, and the counts of all 32
// are computed at once as bit planes (bit b of every cell's count in one
// word), with full adders made of bitwise operations:
//
//   horizontal  h(y, x) = sum_{|d| <= r} cell(y, x + d): the 2r + 1 shifted
//               copies of a row word (funnel shifts with the neighbouring
//               words, fetched by warp shuffles) added as 1-bit numbers;
//   vertical    S(y, x) = sum_{|d| <= r} h(y + d, x): 2r + 1 bit-sliced
//               numbers added (the horizontal sums of a thread's rows are
//               kept in registers while it walks down its strip).
//
// S is the Moore box count with the centre (Sec. IV, Eqs. 1-2 compute the
// same number as band products).  One thread per word column and strip of
// kRows output rows; a warp covers 32 consecutive words of a row.
#include <cuda_runtime.h>

#include <cstdint>

#include "cat_planes.cuh"

namespace cat {
namespace {

constexpr int kRows = 32;        // output rows per thread
constexpr int kBlock = 256;      // threads: 8 warps side by side, 256 words

// Bits needed for a value up to n.
constexpr int bits_for(int n) { return n < 2 ? 1 : 1 + bits_for(n / 2); }

template <int R>
struct Bits {
  static constexpr int kH = bits_for(2 * R + 1);                 // bits of a horizontal sum
  static constexpr int kS = bits_for((2 * R + 1) * (2 * R + 1));  // bits of a box count
};
static_assert(Bits<1>::kH == 2 && Bits<1>::kS == 4 && Bits<2>::kS == 5 && Bits<3>::kS == 6 && Bits<5>::kS == 7,
              "plane counts");

// acc += x (bit-sliced, NX-bit x into an NB-bit accumulator).
template <int NB, int NX>
__device__ __forceinline__ void bs_add(uint32_t (&acc)[NB], const uint32_t (&x)[NX]) {
  uint32_t c = 0;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const uint32_t xb = b < NX ? x[b] : 0u;
    const uint32_t a = acc[b];
    acc[b] = a ^ xb ^ c;
    c = (a & xb) | (c & (a ^ xb));
  }
}

struct SwarParams {
  const uint32_t *in;
  int64_t pitch_words;   // 32-bit words between rows
  int32_t H, W, words;   // rows, cells per row, words holding them
  int32_t *sums;         // counts, or next states
  int64_t sums_ld;
  uint32_t *out;
  uint32_t bound[4][planes::kMaxS];
};

template <int R, bool STEP>
__global__ void __launch_bounds__(kBlock) ltl_swar_kernel(const SwarParams p) {
  constexpr int NH = Bits<R>::kH, NS = Bits<R>::kS, WIN = 2 * R + 1;
  const int lane = threadIdx.x & 31;
  const int wi = blockIdx.x * kBlock + threadIdx.x;             // word column
  const bool col = wi < p.words;
  const int last_bits = p.W - 32 * (p.words - 1);                 // valid bits of the last word
  const uint32_t last_mask = last_bits < 32 ? (1u << last_bits) - 1u : ~0u;
  const uint32_t mask = wi == p.words - 1 ? last_mask : ~0u;
  // the neighbour word this lane loads besides its own: lane 0 the one to the
  // left of the warp, lane 31 the one to the right (a warp covers 32 words)
  const int nc = lane == 0 ? wi - 1 : lane == 31 ? wi + 1 : wi;
  const bool nc_ok = nc >= 0 && nc < p.words;
  const uint32_t nmask = nc == p.words - 1 ? last_mask : ~0u;
  const uint32_t *in_c = p.in + (col ? wi : 0), *in_n = p.in + (nc_ok ? nc : 0);
  if (STEP) {   // (ordinary loads: the launch may start before the grid that it reads is written)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }

  // horizontal sums of row y for this thread's 32 cells (every lane takes part)
  auto hsum = [&](int y, uint32_t (&h)[NH]) {
    const bool row_ok = y >= 0 && y < p.H;
    const int64_t ro = row_ok ? (int64_t)y * p.pitch_words : 0;
    const uint32_t w = (row_ok && col) ? in_c[ro] & mask : 0u;
    const uint32_t x = (row_ok && nc_ok) ? in_n[ro] & nmask : 0u;
    uint32_t left = __shfl_up_sync(0xffffffffu, w, 1), right = __shfl_down_sync(0xffffffffu, w, 1);
    if (lane == 0) left = x;
    if (lane == 31) right = x;
#pragma unroll
    for (int b = 0; b < NH; ++b) h[b] = 0u;
    const uint32_t w1[1] = {w};
    bs_add<NH, 1>(h, w1);
#pragma unroll
    for (int d = 1; d <= R; ++d) {
      const uint32_t l[1] = {__funnelshift_l(left, w, d)};    // cell x - d at bit x
      const uint32_t r[1] = {__funnelshift_r(w, right, d)};   // cell x + d at bit x
      bs_add<NH, 1>(h, l);
      bs_add<NH, 1>(h, r);
    }
  };

  // strips of kRows rows, grid-stride in y (grids taller than 65535 strips)
  for (int64_t y0 = (int64_t)blockIdx.y * kRows; y0 < p.H; y0 += (int64_t)gridDim.y * kRows) {
    uint32_t hs[WIN][NH];
#pragma unroll
    for (int k = 0; k < WIN - 1; ++k) hsum((int)y0 - R + k, hs[k + 1]);
    for (int i = 0; i < kRows; ++i) {
      const int y = (int)y0 + i;
      if (y >= p.H) break;                                        // uniform across the block
#pragma unroll
      for (int k = 0; k < WIN - 1; ++k) {
#pragma unroll
        for (int b = 0; b < NH; ++b) hs[k][b] = hs[k + 1][b];
      }
      hsum(y + R, hs[WIN - 1]);
      uint32_t S[NS];
#pragma unroll
      for (int b = 0; b < NS; ++b) S[b] = b < NH ? hs[0][b] : 0u;
#pragma unroll
      for (int k = 1; k < WIN; ++k) bs_add<NS, NH>(S, hs[k]);
      if (!col) continue;
      if (STEP) {
        const uint32_t c = in_c[(int64_t)y * p.pitch_words];
        const uint32_t keep = planes::at_least<NS>(S, p.bound[planes::kSurviveLo]) & ~planes::at_least<NS>(S, p.bound[planes::kSurviveHi]);
        const uint32_t born = planes::at_least<NS>(S, p.bound[planes::kBirthLo]) & ~planes::at_least<NS>(S, p.bound[planes::kBirthHi]);
        p.out[(int64_t)y * p.pitch_words + wi] = ((c & keep) | (~c & born)) & mask;
        continue;
      }
      int32_t *row = p.sums + (int64_t)y * p.sums_ld;
      for (int t = 0; t < 32 && 32 * wi + t < p.W; ++t) {
        int v = 0;
#pragma unroll
        for (int b = 0; b < NS; ++b) v |= (int)((S[b] >> t) & 1u) << b;
        row[32 * wi + t] = v;
      }
    }
  }
}

typedef void (*SwarKernel)(SwarParams);
template <bool STEP>
SwarKernel swar_kernel(int r) {
  switch (r) {
    case 1: return ltl_swar_kernel<1, STEP>;
    case 2: return ltl_swar_kernel<2, STEP>;
    case 3: return ltl_swar_kernel<3, STEP>;
    case 4: return ltl_swar_kernel<4, STEP>;
    case 5: return ltl_swar_kernel<5, STEP>;
    default: return nullptr;
  }
}

SwarParams swar_params(const uint8_t *in, int64_t pitch, int64_t H, int64_t W) {
  SwarParams p{};
  p.in = reinterpret_cast<const uint32_t *>(in);
  p.pitch_words = pitch / 4;
  p.H = (int32_t)H;
  p.W = (int32_t)W;
  p.words = (int32_t)((W + 31) / 32);
  return p;
}

dim3 swar_grid(const SwarParams &p) {
  const int64_t strips = ((int64_t)p.H + kRows - 1) / kRows;
  return dim3((unsigned)((p.words + kBlock - 1) / kBlock), (unsigned)(strips < 65535 ? strips : 65535));
}

}  // namespace

cudaError_t swar_sums_launch(const uint8_t *in, int64_t pitch, int64_t H, int64_t W, const RuleDev &rule, int32_t *sums,
                             int64_t sums_ld, cudaStream_t s) {
  const SwarKernel kern = swar_kernel<false>(rule.r);
  if (!kern) return cudaErrorInvalidValue;
  SwarParams p = swar_params(in, pitch, H, W);
  p.sums = sums;
  p.sums_ld = sums_ld;
  kern<<<swar_grid(p), kBlock, 0, s>>>(p);
  return cudaGetLastError();
}

cudaError_t swar_step_launch(const PlanesGrid &g, cudaStream_t s) {
  const SwarKernel kern = swar_kernel<true>(g.rule.r);
  if (!kern) return cudaErrorInvalidValue;
  SwarParams p = swar_params(g.in, g.pitch, g.H, g.W);
  p.out = reinterpret_cast<uint32_t *>(g.out);
  planes::set_bounds(p.bound, g.rule, planes::bits_for((2 * g.rule.r + 1) * (2 * g.rule.r + 1)));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = swar_grid(p);
  cfg.blockDim = dim3(kBlock);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace cat
