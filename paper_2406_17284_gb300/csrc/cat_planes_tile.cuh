// Box sums in bit planes on tiles in shared memory, k steps per launch
// (temporal blocking): two states, one bit per cell or uint8 on either side.
//
// The streaming kernel (cat_planes.cuh) first sums 2r rows before a strip's
// first output row, and a launch of it advances one step: on small grids, whose
// strips are short, that start and the launch itself are the time.  Here a
// block of kWarps warps shares the horizontal sums of a strip's rows in shared
// memory (each row's sum is formed once) and advances the strip k steps before
// it is written back, on k r more rows on either side; the words beside the
// strip go stale by r cells a step, which bounds k.  Lanes map to words of a
// virtual row as in the streaming kernel.
#pragma once
#include "cat_planes.cuh"

namespace cat {
namespace planes {

constexpr int kTileWarps = 16;   // (32 warps measured no faster)

struct TileParams {
  Params p;             // p.rows: output rows per strip
  int32_t steps;        // k
  int32_t in_u8, out_u8;
};

template <int R>
__global__ void __launch_bounds__(32 * kTileWarps) planes_tile_kernel(const __grid_constant__ TileParams t) {
  using D = Dim<R>;
  constexpr int NH = D::kH, NS = D::kS, kSlot = 128 * NH, kBlockBytes = 128 * NS;
  extern __shared__ __align__(16) uint8_t smem[];
  const Params &p = t.p;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int halo = t.steps * R, rows = p.rows + 2 * halo;
  uint32_t *cur = reinterpret_cast<uint32_t *>(smem), *nxt = cur + 32 * rows;
  uint8_t *const sums = smem + 256 * rows, *const blocks = sums + kSlot * rows;

  // this lane's strip and word column, as in planes_kernel (no frame)
  const int v = (int)blockIdx.x * kOut + lane - 1;
  int strip = v < 0 ? 0 : v / p.seg;
  int w = v < 0 ? p.seg - 1 : v - strip * p.seg;
  const bool held = w < p.seg - 1 && strip < p.strips;
  w = w < p.seg - 1 ? w : p.seg - 2;
  strip = strip < p.strips ? strip : p.strips - 1;
  const int64_t y0 = (int64_t)strip * p.rows, ys = y0 - halo;   // row i of the tile is grid row ys + i
  const int64_t left = p.W - (int64_t)w * 32;                   // cells from the word's first one on
  const uint32_t mask = !held ? 0u : left >= 32 ? ~0u : (1u << (int)left) - 1u;
  const int lo = ys < 0 ? (int)-ys : 0;                         // rows [lo, hi) of the tile are the grid's
  const int hi = p.H - ys < rows ? (int)(p.H - ys) : rows;
  const uint32_t pitch = (uint32_t)p.pitch;
  const uint8_t *const src = p.in + ys * p.pitch + (int64_t)w * (t.in_u8 ? 32 : 4);
  const uint8_t *const dst = p.out + ys * p.pitch + (int64_t)w * (t.out_u8 ? 32 : 4);
  const bool writes = held && lane >= 1 && lane <= kOut;

  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

#pragma unroll 4
  for (int i = warp; i < rows; i += kTileWarps) {
    uint32_t c = 0u;
    if (i >= lo && i < hi) {
      const uint8_t *q = row_ptr(src, (uint32_t)i, pitch);
      if (t.in_u8) {
        Raw<CAT_STORE_U8> r;
        ld16(r.v, q);
        if (left > 16) {
          ld16(r.v + 4, q + 16);
        } else {
          r.v[4] = r.v[5] = r.v[6] = r.v[7] = 0u;
        }
        if (left < 32) {   // bytes past W belong to whoever owns the buffer
#pragma unroll
          for (int b = 0; b < 8; ++b) {
            const int cells = (int)left - 4 * b;
            r.v[b] &= cells >= 4 ? ~0u : cells <= 0 ? 0u : (1u << (8 * cells)) - 1u;
          }
        }
        c = flags<CAT_STORE_U8, false>(r);
      } else {
        c = *reinterpret_cast<const uint32_t *>(q);
      }
    }
    cur[32 * i + lane] = c & mask;
  }
  __syncthreads();

  // S += h (NX planes)
  auto add = [](auto &S, const auto &h, auto nx) {
    constexpr int NX = decltype(nx)::value;
    uint32_t cy = 0u;
#pragma unroll
    for (int b = 0; b < NS; ++b) {
      const uint32_t a = S[b], x = b < NX ? h[b] : 0u;
      S[b] = a ^ x ^ cy;
      cy = (a & x) | (cy & (a ^ x));
    }
  };
  const std::integral_constant<int, NH> kh{};
  const std::integral_constant<int, NS> ks{};

  for (int s = 1; s <= t.steps; ++s) {
    // Horizontal sums of the rows that this step's output rows reach, a block
    // of consecutive rows per warp, and the blocks' sums.
    const int base = (s - 1) * R, n = rows - 2 * s * R, reach = n + 2 * R;
    const int block = (reach + kTileWarps - 1) / kTileWarps;
    // (with 2r rows before a warp's first output row that cost more than adding
    // up the blocks: 2048^2, r = 16: 7.4 -> 6.1 us a step; r = 4: 2.7 -> 2.9)
    const bool use_blocks = R >= 8 && block > 1 && R >= block;
    {
      const int e = (warp + 1) * block < reach ? (warp + 1) * block : reach;
      uint32_t T[NS];
#pragma unroll
      for (int b = 0; b < NS; ++b) T[b] = 0u;
#pragma unroll 2
      for (int i = warp * block; i < e; ++i) {
        const uint32_t c = cur[32 * (base + i) + lane];
        uint32_t h[NH];
        const uint32_t b = __funnelshift_l(__shfl_up_sync(kFull, c, 1), c, R);
        window_sum<D::kWin, NH>(b, __shfl_down_sync(kFull, b, 1), h);
        ring_store<NH, 32>(sums + (base + i) * kSlot, lane, h);
        if (use_blocks) add(T, h, kh);
      }
      if (use_blocks) ring_store<NS, 32>(blocks + warp * kBlockBytes, lane, T);
    }
    __syncthreads();
    // Each warp takes consecutive output rows: the sum of the 2r rows before
    // the first one's last (whole blocks where they fit), then sliding.
    const int each = (n + kTileWarps - 1) / kTileWarps;
    const int first = s * R + warp * each, end = first + each < rows - s * R ? first + each : rows - s * R;
    uint32_t S[NS];
#pragma unroll
    for (int b = 0; b < NS; ++b) S[b] = 0u;
    if (first < end) {
      auto add_singles = [&](int i, int to) {
#pragma unroll 2
        for (; i < to; ++i) {
          uint32_t h[NH];
          ring_load<NH, 32>(sums + i * kSlot, lane, h);
          add(S, h, kh);
        }
      };
      const int from = first - R, to = first + R;
      if (use_blocks) {
        const int b0 = (from - base + block - 1) / block, b1 = (to - base) / block;
        add_singles(from, base + b0 * block);
        for (int b = b0; b < b1; ++b) {
          uint32_t h[NS];
          ring_load<NS, 32>(blocks + b * kBlockBytes, lane, h);
          add(S, h, ks);
        }
        add_singles(base + b1 * block, to);
      } else {
        add_singles(from, to);
      }
    }
    for (int i = first; i < end; ++i) {
      uint32_t h[NH], o[NH];
      ring_load<NH, 32>(sums + (i + R) * kSlot, lane, h);
#pragma unroll
      for (int b = 0; b < NH; ++b) o[b] = 0u;
      if (i > first) ring_load<NH, 32>(sums + (i - R - 1) * kSlot, lane, o);
      uint32_t br = 0u, cy = 0u;
#pragma unroll
      for (int b = 0; b < NH; ++b) {
        const uint32_t d = h[b] ^ o[b] ^ br;
        br = (~h[b] & o[b]) | (br & ~(h[b] ^ o[b]));
        h[b] = d;
      }
#pragma unroll
      for (int b = 0; b < NS; ++b) {
        const uint32_t a = S[b], x = b < NH ? h[b] : br;
        S[b] = a ^ x ^ cy;
        cy = (a & x) | (cy & (a ^ x));
      }
      const uint32_t c = cur[32 * i + lane];
      const uint32_t keep = at_least<NS>(S, p.bound[kSurviveLo]) & ~at_least<NS>(S, p.bound[kSurviveHi]);
      const uint32_t born = at_least<NS>(S, p.bound[kBirthLo]) & ~at_least<NS>(S, p.bound[kBirthHi]);
      const uint32_t in = ((c & keep) | (~c & born)) & mask;
      if (s < t.steps) {
        nxt[32 * i + lane] = i >= lo && i < hi ? in : 0u;   // cells outside the grid stay dead
      } else if (writes && i < hi) {   // (the output rows start at y0 >= 0)
        uint8_t *q = const_cast<uint8_t *>(row_ptr(dst, (uint32_t)i, pitch));
        if (!t.out_u8) {
          *reinterpret_cast<uint32_t *>(q) = in;
        } else {
          uint32_t a[4], e[4];
          const uint32_t lo4 = in & 0x0F0F0F0Fu, hi4 = (in >> 4) & 0x0F0F0F0Fu;
          spread_bytes<0>(lo4, hi4, a);
          spread_bytes<1>(lo4, hi4, e);
          if (left >= 16) *reinterpret_cast<uint4 *>(q) = make_uint4(a[0], a[1], a[2], a[3]);
          else store_part(q, a, (int)left);
          if (left >= 32) *reinterpret_cast<uint4 *>(q + 16) = make_uint4(e[0], e[1], e[2], e[3]);
          else if (left > 16) store_part(q + 16, e, (int)left - 16);
        }
      }
    }
    __syncthreads();
    uint32_t *const swap = cur;
    cur = nxt;
    nxt = swap;
  }
}

struct TileKernel {
  void (*fn)(TileParams) = nullptr;
  int row_bytes = 0, block_bytes = 0, planes = 0;   // shared memory per row of the tile, for the blocks' sums
};
TileKernel tile_kernel(int r);   // r <= kMaxR

template <int LO = 1>
TileKernel find_tile_kernel(int r) {
  if constexpr (LO > kMaxR) {
    return TileKernel{};
  } else {
    if (r == LO) return TileKernel{planes_tile_kernel<LO>, 128 * (2 + Dim<LO>::kH), 128 * Dim<LO>::kS * kTileWarps, Dim<LO>::kS};
    return find_tile_kernel<LO + 1>(r);
  }
}

}  // namespace planes
}  // namespace cat
