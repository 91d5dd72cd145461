// Periodic boundary: the ghost frame.
//
// A periodic instance keeps its H x W grid inside a frame of G = 16 ghost cells
// on every side (G >= r for every served radius).  Before each step this kernel
// writes every ghost cell with the grid cell it wraps to, ((y mod H), (x mod W))
// in grid coordinates, so the step kernel can treat the framed grid like any
// other: its windows read real neighbours across every edge (the paper's own
// boundary, Sec. V), and its tiles start at TMA coordinate (x0 + G, y0 + G),
// which keeps every TMA x-coordinate 16-byte aligned.  The frame is 2G(W + 2G)
// + 2GH cells: 1.05 M cells for a 16384^2 grid, against 268 M in the grid.
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "cat_internal.h"

namespace cat {
namespace {

__device__ __forceinline__ int wrap32(int v, int n) {
  v %= n;
  return v < 0 ? v + n : v;
}

// The frame in three kinds of items, none of which reads a ghost cell, so
// they need no order among themselves:
//   rows     the grid columns of the 2G frame rows, 16 bytes per item (the
//            framed row and its source share the offset G = 16, so full
//            chunks are aligned 16-byte copies);
//   columns  the G left and G right frame cells of one grid row (two aligned
//            16-byte copies when W is a multiple of 16, else per byte);
//   corners  the 4 G x G corner cells, one per item.
// Grid-stride over rows, then columns, then corners.  The kernel lets the
// next kernel in the stream start its set-up and reads the grid only after
// the previous kernel (the step that wrote it) has completed.
__global__ void ghost_fill_kernel(uint8_t *base, int64_t pitch, int H, int W, int G) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int chunks = (W + 15) / 16;
  const int64_t n_rows = 2 * (int64_t)G * chunks, n_cols = 2 * (int64_t)H, n_corners = 4 * (int64_t)G * G;
  const int64_t n_all = n_rows + n_cols + n_corners;
  const bool vec_cols = (W % 16) == 0 && W >= G;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_all; i += (int64_t)gridDim.x * blockDim.x) {
    if (i < n_rows) {
      const int fr = (int)(i / chunks), ch = (int)(i - (int64_t)fr * chunks);
      const int py = fr < G ? fr : H + fr;                       // rows 0..G-1 and H+G..H+2G-1
      const int sy = wrap32(py - G, H) + G;
      uint8_t *dst = base + (int64_t)py * pitch + G + 16 * ch;
      const uint8_t *src = base + (int64_t)sy * pitch + G + 16 * ch;
      if (16 * ch + 16 <= W) {
        *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(src);
      } else {
        for (int b = 0; b < W - 16 * ch; ++b) dst[b] = src[b];
      }
    } else if (i < n_rows + n_cols) {
      const int64_t k = i - n_rows;
      const int y = (int)(k >> 1), side = (int)(k & 1);
      uint8_t *row = base + (int64_t)(G + y) * pitch;
      const int px0 = side ? W + G : 0;                          // first frame column of this side
      if (vec_cols && G == 16) {
        // left: grid columns W-16..W-1 (framed W..W+15); right: grid 0..15 (framed 16..31)
        *reinterpret_cast<uint4 *>(row + px0) = *reinterpret_cast<const uint4 *>(row + (side ? G : W));
      } else {
        for (int b = 0; b < G; ++b) row[px0 + b] = row[wrap32(px0 + b - G, W) + G];
      }
    } else {
      const int k = (int)(i - n_rows - n_cols), corner = k / (G * G), c = k - corner * G * G;
      const int py = (corner & 1 ? H + G : 0) + c / G, px = (corner & 2 ? W + G : 0) + c % G;
      base[(int64_t)py * pitch + px] = base[(int64_t)(wrap32(py - G, H) + G) * pitch + wrap32(px - G, W) + G];
    }
  }
}

// The same for H, W >= 16 and below 2^19 rows, which is nearly every grid, in as few instructions
// as that takes, a thread per cell: frame position f of 32 (0 .. 15 before the
// grid, 16 .. 31 after it) is framed coordinate f or N + f and wraps to N + f
// or f.  The step kernel leaves none of these instructions in an SM's cache,
// so their number is the kernel's time: loops over a thread's cells and a
// remainder for each (above) took longer than the step itself where W % 16 is
// not 0, and whole chunks shifted into place in registers hardly less
// (4600^2, r = 5, tensor-core steps back to back: 64 and 31 us a step; so
// 14.8, and 13.1 with no frame to refresh).
// CHUNKS: a thread takes 16 cells of the sides (W % 16 = 0, so both ends are
// aligned).  Tall grids need it, whose sides are the work: r = 12, a thread per
// cell / per chunk, 16384 x 64 8.0 / 7.1 us a step, 65536 x 64 17.8 / 12.0,
// 1048576 x 64 206 / 103, 131072 x 256 34.5 / 22.3; others gain nothing (8192 x
// 1024 9.9 / 9.9, 16384 x 4096 34.2 / 33.7 and at r = 5 33.2 / 33.8).  From 2^19
// rows on the loop above is as fast or, where the grid is about as large as the
// L2, faster (r = 4, loop / chunks: 524288 x 128 53.7 / 53.1, 700000 x 128 73.9 /
// 79.6, 819200 x 128 87 / 97, 1638400 x 128 191.8 / 190.3).
// early: the next kernel may start its set-up beside the previous one's end.
// The tensor-core step gains by that (256^2: 5.6 against 6.4), the bit-plane
// steps, whose blocks only wait, lose (2048^2, r = 12, two steps: 10.1 against 9.1).
__device__ __forceinline__ int frame_at(int f, int n) { return f < 16 ? f : n + f; }
__device__ __forceinline__ int frame_from(int f, int n) { return f < 16 ? n + f : f; }

template <bool CHUNKS>
__global__ void ghost_frame_kernel(uint8_t *base, int64_t pitch, int H, int W, unsigned row_blocks, bool early) {
  if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (!early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (blockIdx.x < row_blocks) {   // the grid's columns of the 32 frame rows: chunks of 16, then single cells
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x, chunks = (unsigned)W / 16, per = chunks + W % 16;
    const unsigned f = i / per, k = i - f * per;
    if (f >= 32) return;
    uint8_t *dst = base + frame_at((int)f, H) * pitch + 16;
    const uint8_t *src = base + frame_from((int)f, H) * pitch + 16;
    if (k < chunks) reinterpret_cast<uint4 *>(dst)[k] = reinterpret_cast<const uint4 *>(src)[k];
    else dst[15 * (int64_t)chunks + k] = src[15 * (int64_t)chunks + k];
  } else {                         // the frame's cells beside the grid's rows, and the corners
    const int64_t i = (int64_t)(blockIdx.x - row_blocks) * blockDim.x + threadIdx.x, q = CHUNKS ? i >> 1 : i >> 5;
    if (q >= H + 32) return;
    const int f = CHUNKS ? 16 * (int)(i & 1) : (int)(i & 31);
    const int64_t to = q < H ? q + 16 : frame_at((int)(q - H), H), from = q < H ? q + 16 : frame_from((int)(q - H), H);
    uint8_t *const dst = base + to * pitch + frame_at(f, W);
    const uint8_t *const src = base + from * pitch + frame_from(f, W);
    if (CHUNKS) *reinterpret_cast<uint4 *>(dst) = *reinterpret_cast<const uint4 *>(src);
    else *dst = *src;
  }
}

// The ghost frame of a one-bit grid (the states between the steps of one call):
// position p of a row holds cell p - 16, so the grid's cells start in the middle
// of word 0 and the frame's right cells end the row.  Items, again in few
// instructions: the words with cells beside the grid's columns, a thread per
// row of the frame, and the other words of the 32 frame rows; each made from
// its source row's grid cells only.
__global__ void ghost_bits_kernel(uint32_t *base, int64_t pitch_words, int H, int W, int words, unsigned row_blocks) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int wr = (W + 16) / 32;                        // cells W .. W + 15 start in this word
  const bool middle = blockIdx.x < row_blocks;
  int64_t q = (int64_t)(blockIdx.x - (middle ? 0u : row_blocks)) * blockDim.x + threadIdx.x;
  int w = 0;
  if (middle) {
    const unsigned k = (unsigned)q / (unsigned)words;
    w = (int)((unsigned)q - k * (unsigned)words);
    q = H + k;
    if (w == 0 || w >= wr) return;
  }
  if (q >= H + 32) return;
  const int f = (int)(q - H);
  const int row = f < 0 ? (int)q : f < 16 ? f - 16 : H + f - 16;
  const uint32_t *src = base + (f < 0 ? row : wrap32(row, H)) * pitch_words;
  uint32_t *dst = base + row * pitch_words;
  if (middle) {
    dst[w] = src[w];
    return;
  }
  const int sl = W % 32, sr = (W + 16) % 32;
  const uint32_t first = src[0], right = first >> 16;
  const uint32_t left = __funnelshift_r(src[W / 32], src[W / 32 + 1], sl) & 0xFFFFu;   // cells W - 16 .. W - 1
  const uint32_t last = (src[wr] & ((1u << sr) - 1u)) | (right << sr);                 // the grid's last cells, then the frame's
  dst[0] = (first & 0xFFFF0000u) | left;
  dst[wr] = last;
  if (wr + 1 < words) dst[wr + 1] = sr > 16 ? right >> (32 - sr) : 0u;
}

}  // namespace

cudaError_t ghost_prepare(int device) {
  static std::atomic<uint32_t> loaded{0};   // by device
  const uint32_t bit = device >= 0 && device < 32 ? 1u << device : 0u;
  if (loaded.load(std::memory_order_relaxed) & bit) return cudaSuccess;
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, ghost_fill_kernel);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, ghost_frame_kernel<false>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, ghost_frame_kernel<true>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, ghost_bits_kernel);
  if (e == cudaSuccess) loaded.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

cudaError_t ghost_bits_launch(uint8_t *row0, int64_t pitch, int64_t H, int64_t W, cudaStream_t s) {
  const int words = (int)((W + 32 + 31) / 32), threads = 256;
  const int64_t rows = (32 * (int64_t)words + threads - 1) / threads, sides = (H + 32 + threads - 1) / threads;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(rows + sides));
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ghost_bits_kernel, reinterpret_cast<uint32_t *>(row0), pitch / 4, (int)H, (int)W,
                            words, (unsigned)rows);
}

// Launched programmatically dependent on the previous kernel in the stream
// (see ghost_fill_kernel); the tcgen05 step launched after it is in turn
// dependent on it.
cudaError_t ghost_fill_launch(uint8_t *base, int64_t pitch, int64_t H, int64_t W, int G, bool early, cudaStream_t s) {
  const int threads = 256;
  const bool chunks = W % 16 == 0 && H >= 16384 && H >= 8 * W;
  const bool loop = H < 16 || W < 16 || G != 16 || (chunks && H >= 1 << 19);
  const int64_t rows = (32 * (W / 16 + W % 16) + threads - 1) / threads;
  const int64_t sides = ((H + 32) * (chunks ? 2 : 32) + threads - 1) / threads;
  const int64_t n = 2 * (int64_t)G * ((W + 15) / 16) + 2 * H + 4 * (int64_t)G * G;
  const int64_t want = (n + threads - 1) / threads;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(!loop ? rows + sides : want < 4096 ? want : 4096));
  cfg.blockDim = dim3(threads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (loop) return cudaLaunchKernelEx(&cfg, ghost_fill_kernel, base, pitch, (int)H, (int)W, G);
  return cudaLaunchKernelEx(&cfg, chunks ? ghost_frame_kernel<true> : ghost_frame_kernel<false>, base, pitch, (int)H, (int)W,
                            (unsigned)rows, early);
}

}  // namespace cat
