// Box sums in bit planes: the step kernel body shared by the translation
// units cat_planes_*.cu (one storage each, so that they compile in parallel).
//
// A thread owns 32 consecutive cells of a row (one word of flags [state == 1])
// and walks down a strip of rows.  A number per cell is held as bit planes
// (bit b of all 32 numbers in one word), so one three-input logic operation
// adds one bit of 32 cells:
//
//   horizontal  h(x) = sum_{d = 0..2r} cell(x - r + d), by halving: a window
//               of 2m (+ 1) cells is two windows of m cells, the second
//               shifted by m, (plus one cell as the carry-in).  The planes of
//               the cells to the right come from the next lane by shuffle, so
//               the cost is about 5 log2(2r) operations for any r;
//   vertical    S(y) = S(y - 1) + h(y + r) - h(y - r - 1): the last 2r + 1
//               horizontal sums of each thread stay in a ring in shared
//               memory, so the cost does not grow with r either;
//   rule        S >= K for the four bounds of the reduced rule, each the carry
//               chain of a bit-sliced subtraction; the centre cell picks the
//               survival or the birth range.
//
// All additions are exact, so the next states are those of every other kernel
// (Sec. IV, Eqs. 1-2 define the same count as two band products).
//
// What bounds it: the integer pipe (ncu, 16384^2: one bit per cell, r = 2 / 16:
// ALU 78% / 83%, DRAM 10% / 5%; C = 16, r = 10: four bits 81%, one byte 74%).
// 32768^2 one-bit steps: r = 2 224 -> 148 us, r = 16 594 -> 327 us; 24576^2,
// C = 16, r = 10: four bits 435 -> 269 us, one byte 398 -> 333 us (before: the
// tensor-core kernels, and at r <= 5 a bit-sliced kernel that added the 2r + 1
// cells and rows one by one).
//
// Lanes are laid over a virtual row of words: the row strips of the grid side
// by side, each followed by one zero word (the dead cells beyond its right
// edge, which are also the dead cells left of the next strip).  A warp takes
// 32 consecutive virtual words and writes all but the first and the last,
// whose neighbours it does not hold; narrow grids thus fill warps as well as
// wide ones.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "cat_internal.h"

namespace cat {
namespace planes {

// Bits needed for a value up to n.
__host__ __device__ constexpr int bits_for(int n) { return n < 2 ? 1 : 1 + bits_for(n / 2); }

template <int R>
struct Dim {
  static constexpr int kH = bits_for(2 * R + 1);                  // planes of a horizontal sum
  static constexpr int kS = bits_for((2 * R + 1) * (2 * R + 1));  // planes of a box count
  static constexpr int kWin = 2 * R + 1;
  static constexpr int kThreadBytes = 4 * (kH * kWin + R);   // rings of horizontal sums and of centre words
};

constexpr uint32_t kFull = 0xffffffffu;
constexpr int kMaxR = 16;   // a window reaches one word to either side
constexpr int kOut = 30;    // words a warp writes: all but the first and the last

// 32 cells of a row as loaded.
template <int ST>
struct Raw {
  static constexpr int kBytes = ST == CAT_STORE_U8 ? 32 : ST == CAT_STORE_NIB4 ? 16 : 4;
  static constexpr int kWords = kBytes / 4;
  uint32_t v[kWords];
};

// Ordinary loads: a programmatically dependent launch starts before the grid
// it reads is written, so the read-only path must not be used.
__device__ __forceinline__ void ld16(uint32_t *v, const uint8_t *p) {
  const uint4 a = *reinterpret_cast<const uint4 *>(p);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}

// State-1 flags of 32 loaded cells: bit x = [cell x is 1].
// uint8, two states: four cells' 0/1 bytes are combined pairwise (w | w' << 4)
// and the eight flags gathered into the top byte by one multiplication whose
// partial products never meet (all on the multiply pipe; three byte permutes
// join the four bytes).
template <int ST, bool MS>
__device__ __forceinline__ uint32_t flags(const Raw<ST> &r) {
  if constexpr (ST == CAT_STORE_BIT1) {
    return r.v[0];
  } else {
    uint32_t q[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if constexpr (ST == CAT_STORE_U8 && !MS) {
        const uint32_t t = r.v[2 * j + 1] * 16u + r.v[2 * j];
        q[j] = t * 0x01020408u;
      } else {
        const uint32_t t = ST == CAT_STORE_U8 ? r.v[(2 * j + 1) & 7] * 16u + r.v[(2 * j) & 7] : r.v[j & 3];
        // bit 3 of a nibble of f: the state is 1 (t ^ 1 is zero; no nibble carries)
        const uint32_t x = t ^ 0x11111111u;
        const uint32_t f = ~(((x & 0x77777777u) + 0x77777777u) | x) & 0x88888888u;
        if constexpr (ST == CAT_STORE_U8) q[j] = f * 0x00204081u;              // nibble order: cells 0,4,1,5,2,6,3,7
        else q[j] = ((f | (f >> 3)) & 0x18181818u) * 0x00208208u;             // nibble order: cells 0..7
      }
    }
    return __byte_perm(__byte_perm(q[0], q[1], 0x0073), __byte_perm(q[2], q[3], 0x0073), 0x5410);
  }
}

// b(x + D) of a plane for the cell x at bit x, D in 1..32 (next: the plane in
// the next lane).
template <int D>
__device__ __forceinline__ uint32_t shift_right(uint32_t own, uint32_t next) {
  if constexpr (D < 32) return __funnelshift_r(own, next, D);
  else return next;
}

// Window sums of M cells to the right of each cell (M cells starting at it):
// planes h[0 .. bits_for(M)).
template <int M, int NH>
__device__ __forceinline__ void window_sum(uint32_t b, uint32_t next, uint32_t (&h)[NH]) {
  if constexpr (M == 1) {
    h[0] = b;
  } else {
    constexpr int HM = M / 2, NB = bits_for(HM), NO = bits_for(M);
    window_sum<HM, NH>(b, next, h);
    uint32_t c = 0u;
    if constexpr (M & 1) c = shift_right<2 * HM>(b, next);
    uint32_t o[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      if constexpr (HM == 1) o[i] = shift_right<1>(b, next);
      else o[i] = shift_right<HM>(h[i], __shfl_down_sync(kFull, h[i], 1));
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const uint32_t a = h[i];
      h[i] = a ^ o[i] ^ c;
      c = (a & o[i]) | (c & (a ^ o[i]));
    }
    if constexpr (NO > NB) h[NB] = c;
  }
}

// S >= K for every cell: the carry out of S + ~K + 1, one majority function
// per plane; k[i] is bit i of ~K over a whole word (kernel parameters, so the
// words are constant operands).
template <int NS>
__device__ __forceinline__ uint32_t at_least(const uint32_t (&S)[NS], const uint32_t *k) {
  uint32_t c = S[0] | k[0];
#pragma unroll
  for (int i = 1; i < NS; ++i) c = (S[i] & k[i]) | (c & (S[i] | k[i]));
  return c;
}

// Byte j of x in a word of its own.
template <int J>
__device__ __forceinline__ uint32_t byte_of(uint32_t x) { return __byte_perm(x, 0u, 0x4440 + J); }

// 16 flags (bytes 2 T and 2 T + 1 of a word whose low and high nibbles are the
// bytes of lo and hi) -> four words of four 0/1 bytes: a nibble times 2^0 +
// 2^7 + 2^14 + 2^21 has bit i at bit 8 i (the copies do not overlap).
template <int T>
__device__ __forceinline__ void spread_bytes(uint32_t lo, uint32_t hi, uint32_t (&o)[4]) {
  o[0] = (byte_of<2 * T>(lo) * 0x00204081u) & 0x01010101u;
  o[1] = (byte_of<2 * T>(hi) * 0x00204081u) & 0x01010101u;
  o[2] = (byte_of<2 * T + 1>(lo) * 0x00204081u) & 0x01010101u;
  o[3] = (byte_of<2 * T + 1>(hi) * 0x00204081u) & 0x01010101u;
}

// The first `cells` (< 16) of 16 bytes: those past W are not the grid's.
__device__ __forceinline__ void store_part(uint8_t *q, uint32_t (&a)[4], int cells) {
  if (cells & 8) {
    *reinterpret_cast<uint2 *>(q) = make_uint2(a[0], a[1]);
    q += 8;
    a[0] = a[2]; a[1] = a[3];
  }
  if (cells & 4) {
    *reinterpret_cast<uint32_t *>(q) = a[0];
    q += 4;
    a[0] = a[1];
  }
  if (cells & 2) {
    *reinterpret_cast<uint16_t *>(q) = (uint16_t)a[0];
    q += 2;
    a[0] >>= 16;
  }
  if (cells & 1) *q = (uint8_t)a[0];
}

// Eight flags (a byte) -> eight nibbles 0/1, flag i in nibble i.
__device__ __forceinline__ uint32_t spread_nibbles(uint32_t b) {
  uint32_t x = (b * 0x1001u) & 0x000F000Fu;
  x = (x * 0x41u) & 0x03030303u;
  return (x * 9u) & 0x11111111u;
}

// Next states of eight cells in nibbles: t their states (below C <= 16), f the
// flags (bit 0) of the cells whose count is in range.  State 0 -> f; 1 -> 1 or
// 2 (0 when C = 2, via two = 0); c >= 2 -> c + 1, 0 past C - 1.
__device__ __forceinline__ uint32_t age_nibbles(uint32_t t, uint32_t f, uint32_t last, uint32_t two) {
  const uint32_t u = (t & 0x77777777u) + 0x66666666u;
  const uint32_t g = (u | t) & 0x88888888u;                        // state >= 2
  const uint32_t x = t ^ last;                                     // zero for state C - 1
  const uint32_t k1 = (g & (((x & 0x77777777u) + 0x77777777u) | x)) >> 3;   // 2 <= state < C - 1
  const uint32_t older = (t + k1) & (k1 * 15u);
  const uint32_t g1 = g >> 3;
  const uint32_t lost = (t & two & ~g1) & ~f;                      // state 1, not kept
  return older | (lost * 2u + (f & ~g1));
}

// The ring of horizontal sums, per slot, groups of four planes as 16-byte
// words per thread, then two, then one (conflict-free, few instructions).
template <int NH, int NT>
__device__ __forceinline__ void ring_load(const uint8_t *s, int tid, uint32_t (&h)[NH]) {
  constexpr int G = NH / 4;
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const uint4 a = *reinterpret_cast<const uint4 *>(s + NT * 16 * g + tid * 16);
    h[4 * g] = a.x; h[4 * g + 1] = a.y; h[4 * g + 2] = a.z; h[4 * g + 3] = a.w;
  }
  if constexpr (NH & 2) {
    const uint2 a = *reinterpret_cast<const uint2 *>(s + NT * 16 * G + tid * 8);
    h[4 * G] = a.x; h[4 * G + 1] = a.y;
  }
  if constexpr (NH & 1) h[NH - 1] = *reinterpret_cast<const uint32_t *>(s + NT * 4 * (NH - 1) + tid * 4);
}
template <int NH, int NT>
__device__ __forceinline__ void ring_store(uint8_t *s, int tid, const uint32_t (&h)[NH]) {
  constexpr int G = NH / 4;
#pragma unroll
  for (int g = 0; g < G; ++g)
    *reinterpret_cast<uint4 *>(s + NT * 16 * g + tid * 16) =
        make_uint4(h[4 * g], h[4 * g + 1], h[4 * g + 2], h[4 * g + 3]);
  if constexpr (NH & 2) *reinterpret_cast<uint2 *>(s + NT * 16 * G + tid * 8) = make_uint2(h[4 * G], h[4 * G + 1]);
  if constexpr (NH & 1) *reinterpret_cast<uint32_t *>(s + NT * 4 * (NH - 1) + tid * 4) = h[NH - 1];
}

constexpr int kMaxS = bits_for((2 * kMaxR + 1) * (2 * kMaxR + 1));
enum { kSurviveLo, kSurviveHi, kBirthLo, kBirthHi };   // in range: >= lo and not >= hi

void set_bounds(uint32_t (*bound)[kMaxS], const RuleDev &rule, int planes);

struct Params {
  const uint8_t *in;   // row 0: cell 0 of the grid for uint8, cell -frame for packed rows
  uint8_t *out;
  int64_t pitch;
  int32_t H, W;
  int32_t written;     // cells written per row (W, or more where what lies past W is not kept)
  int32_t seg;         // words of a strip in the virtual row (the last one is the zero word)
  int32_t rows;        // rows per strip (a multiple of the rows loaded ahead)
  int32_t strips;
  int32_t frame;       // readable cells around the grid (a periodic grid's ghost frame), else 0
  uint32_t last;       // C - 1 in every nibble
  uint32_t two;        // 1 in every nibble when a state-1 cell that fails survival becomes 2, else 0
  uint32_t bound[4][kMaxS];
};

// What a warp holds and how far ahead it loads.
template <int R, bool MS>
struct Cfg {
  static constexpr int kSmem = 32 * Dim<R>::kThreadBytes;
  static constexpr int kBySmem = 232448 / (kSmem + 1024);
  static constexpr int kWarps = kBySmem < 16 ? kBySmem : 16;   // resident warps aimed at
  static constexpr int kAhead = MS ? 2 : 4;   // (the loop body is unrolled as far: larger ones miss the instruction cache)
};

__device__ __forceinline__ const uint8_t *row_ptr(const uint8_t *base, uint32_t row, uint32_t pitch) {
  uint64_t r;   // one multiply-add, off the integer pipe that the adders use
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(row), "r"(pitch), "l"(base));
  return reinterpret_cast<const uint8_t *>(r);
}

// What a lane reads and writes in memory: a 16-cell half of a word (uint8) or a word.
struct Source {
  const uint8_t *base;   // row 0 of its strip's rows
  int lo, hi;            // rows that exist
  int cells;             // uint8: readable cells of the 16
};
struct Target {
  const uint8_t *base;   // output row 0
  int rows;              // rows written
  int cells;             // uint8: cells of the 16 that are the grid's
};

// One step from storage SI to storage SO (the same one, or between uint8 and
// one bit for two states), by one warp; block: which 30 virtual words, smem:
// its rings.
template <int R, int SI, int SO, bool MS, int A = Cfg<R, MS>::kAhead>
__device__ __forceinline__ void planes_step(const Params &p, int block, uint8_t *smem) {
  using D = Dim<R>;
  constexpr int NH = D::kH, NS = D::kS, NT = 32;
  constexpr int kParts = SI == CAT_STORE_U8 ? 2 : 1, kOutParts = SO == CAT_STORE_U8 ? 2 : 1;
  constexpr int kSlot = NT * 4 * NH, kRing = D::kWin * kSlot, kCentre = NT * 4 * R;
  uint8_t *const cring = smem + kRing;
  const int lane = threadIdx.x & 31;

  // this lane's strip and word column (word w holds cells x0 .. x0 + 31); a
  // lane without a word reads along with a neighbour and masks its flags
  const int v = block * kOut + lane - 1;
  int strip = v < 0 ? 0 : v / p.seg;
  int w = v < 0 ? p.seg - 1 : v - strip * p.seg;
  const bool held = w < p.seg - 1 && strip < p.strips;
  w = w < p.seg - 1 ? w : p.seg - 2;
  strip = strip < p.strips ? strip : p.strips - 1;
  const int64_t y0 = (int64_t)strip * p.rows;
  const int64_t x0 = (int64_t)w * 32 - p.frame;
  const int64_t left = p.W + p.frame - x0;   // readable cells from x0 on
  const uint32_t mask = !held ? 0u : left >= 32 ? ~0u : (1u << (int)left) - 1u;
  const int64_t out_left = left + p.written - p.W;   // (packed) cells written from x0 on
  const uint32_t out_mask = SO == CAT_STORE_U8 || out_left >= 32 ? ~0u : (1u << (int)out_left) - 1u;
  const bool writes = held && lane >= 1 && lane <= kOut;
  const int my_rows = !writes ? 0 : p.H - y0 < p.rows ? (int)(p.H - y0) : p.rows;
  // bytes from the row's start: cell 0 of the grid for uint8, cell -frame for packed rows
  const int64_t col_in = (int64_t)w * Raw<SI>::kBytes - (SI == CAT_STORE_U8 ? p.frame : 0);
  const int64_t col_out = (int64_t)w * Raw<SO>::kBytes - (SO == CAT_STORE_U8 ? p.frame : 0);
  // the strip's rows y0 - R + i, i in [0, 2 R + rows); those in [lo, hi) exist
  const int64_t ys = y0 - R;
  const int lo = ys < -p.frame ? (int)(-p.frame - ys) : 0;
  const int hi = (int)(p.H + p.frame - ys < (1 << 30) ? p.H + p.frame - ys : (1 << 30));
  const bool inside = __all_sync(kFull, lo == 0 && hi >= 2 * R + p.rows + A && p.H - y0 >= p.rows);
  const uint32_t pitch = (uint32_t)p.pitch;
  // Memory accesses: one word per lane, or with one byte per cell two 16-cell
  // halves of words, so that a warp's access is contiguous: lane l takes half
  // l & 1 of the words of lanes l / 2 and 16 + l / 2.
  Source from[kParts];
  Target to[kOutParts];
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    if (t < kParts) {
      const int of = kParts == 1 ? lane : 16 * t + (lane >> 1), half = kParts == 1 ? 0 : 16 * (lane & 1);
      const int64_t y = __shfl_sync(kFull, y0, of), c = __shfl_sync(kFull, col_in, of) + half;
      const int64_t readable = __shfl_sync(kFull, left, of) - half;
      from[t].cells = readable >= 16 ? 16 : readable <= 0 ? 0 : (int)readable;
      // (a half without a cell reads the other half, and clears it)
      from[t].base = p.in + (y - R) * p.pitch + c - (readable <= 0 ? 16 : 0);
      from[t].lo = __shfl_sync(kFull, lo, of);
      from[t].hi = __shfl_sync(kFull, hi, of);
    }
    if (t < kOutParts) {
      const int of = kOutParts == 1 ? lane : 16 * t + (lane >> 1), half = kOutParts == 1 ? 0 : 16 * (lane & 1);
      const int64_t x = __shfl_sync(kFull, x0, of) + half, y = __shfl_sync(kFull, y0, of);
      to[t].base = p.out + y * p.pitch + __shfl_sync(kFull, col_out, of) + half;
      to[t].cells = p.written - x >= 16 ? 16 : (int)(p.written - x);
      to[t].rows = __shfl_sync(kFull, my_rows, of);
      if (SO == CAT_STORE_U8 && (x < 0 || x >= p.written)) to[t].rows = 0;
    }
  }
  // some access of the warp ends within its 16 cells
  const bool odd_in = SI == CAT_STORE_U8 && __any_sync(kFull, from[0].cells < 16 || from[kParts - 1].cells < 16);
  const bool odd_out = SO == CAT_STORE_U8 && __any_sync(kFull, to[0].cells < 16 || to[kOutParts - 1].cells < 16);

  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // uint8: bytes past the last readable cell belong to whoever owns the buffer
  uint32_t past[Raw<SI>::kWords];
#pragma unroll
  for (int i = 0; i < Raw<SI>::kWords; ++i) {
    const int cells = from[i / 4 % kParts].cells - 4 * (i % 4);
    past[i] = cells >= 4 ? ~0u : cells <= 0 ? 0u : (1u << (8 * cells)) - 1u;
  }
  auto clear_past = [&](Raw<SI> &r) {
#pragma unroll
    for (int i = 0; i < Raw<SI>::kWords; ++i) r.v[i] &= past[i];
  };
  // flags of a loaded row: uint8, the halves of a lane's word come from lanes
  // 2 l and 2 l + 1, their first accesses for lanes below 16, else their second
  const uint32_t halves = lane < 16 ? 0x5410u : 0x7632u;
  auto flags_of = [&](Raw<SI> r, uint32_t valid) {
    if (odd_in) clear_past(r);
    uint32_t f = flags<SI, MS>(r);
    if constexpr (SI == CAT_STORE_U8)
      f = __byte_perm(__shfl_sync(kFull, f, 2 * lane), __shfl_sync(kFull, f, 2 * lane + 1), halves);
    return f & valid;
  };
  auto hsum = [&](uint32_t c, uint32_t (&h)[NH]) {
    const uint32_t b = __funnelshift_l(__shfl_up_sync(kFull, c, 1), c, R);   // bit x: cell x - R
    window_sum<D::kWin, NH>(b, __shfl_down_sync(kFull, b, 1), h);
  };
  auto next_slot = [&](int &q) {
    const int now = q;
    q = q + kSlot == kRing ? 0 : q + kSlot;
    return now;
  };
  auto next_cslot = [&](int &q) {
    const int now = q;
    q = q + 4 * NT == kCentre ? 0 : q + 4 * NT;
    return now;
  };
  // S += h
  auto add_rows = [&](uint32_t (&S)[NS], const uint32_t (&h)[NH]) {
    uint32_t cy = 0u;
#pragma unroll
    for (int b = 0; b < NS; ++b) {
      const uint32_t a = S[b], x = b < NH ? h[b] : 0u;
      S[b] = a ^ x ^ cy;
      cy = (a & x) | (cy & (a ^ x));
    }
  };
  // S += h - o: the difference (two's complement, its sign in br), then the sum
  auto slide = [&](uint32_t (&S)[NS], uint32_t (&h)[NH], const uint32_t (&o)[NH]) {
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
  };
  auto rule = [&](const uint32_t (&S)[NS], uint32_t centre) {
    const uint32_t keep = at_least<NS>(S, p.bound[kSurviveLo]) & ~at_least<NS>(S, p.bound[kSurviveHi]);
    const uint32_t born = at_least<NS>(S, p.bound[kBirthLo]) & ~at_least<NS>(S, p.bound[kBirthHi]);
    return (centre & keep) | (~centre & born);
  };
  // uint8: flags of the two halves of words that this lane writes
  const uint32_t mine = lane & 1 ? 0x7632u : 0x5410u;
  auto split = [&](uint32_t in) {
    return __byte_perm(__shfl_sync(kFull, in, lane >> 1), __shfl_sync(kFull, in, 16 + (lane >> 1)), mine);
  };
  auto put = [&](int j, uint32_t in, const Raw<SI> &cs) {   // output row j of the strip
    uint32_t lo4 = 0u, hi4 = 0u;
    if constexpr (SO == CAT_STORE_U8) {
      in = split(in);
      lo4 = in & 0x0F0F0F0Fu;
      hi4 = (in >> 4) & 0x0F0F0F0Fu;
    }
#pragma unroll
    for (int t = 0; t < kOutParts; ++t) {
      if (j >= to[t].rows) continue;
      uint8_t *const q = const_cast<uint8_t *>(row_ptr(to[t].base, (uint32_t)j, pitch));
      if constexpr (SO == CAT_STORE_BIT1) {
        *reinterpret_cast<uint32_t *>(q) = in & out_mask;
      } else if constexpr (SO == CAT_STORE_NIB4) {
        const uint32_t f = in & out_mask;
        uint4 a;
        a.x = age_nibbles(cs.v[0], spread_nibbles(byte_of<0>(f)), p.last, p.two);
        a.y = age_nibbles(cs.v[1], spread_nibbles(byte_of<1>(f)), p.last, p.two);
        a.z = age_nibbles(cs.v[2], spread_nibbles(byte_of<2>(f)), p.last, p.two);
        a.w = age_nibbles(cs.v[3], spread_nibbles(byte_of<3>(f)), p.last, p.two);
        *reinterpret_cast<uint4 *>(q) = a;
      } else {
        uint32_t a[4];
        if (t == 0) spread_bytes<0>(lo4, hi4, a);
        else spread_bytes<1>(lo4, hi4, a);
        if constexpr (MS) {
#pragma unroll
          for (int i = 0; i < 2; ++i) {   // nibble pairs: even words in the low nibbles
            const uint32_t u = cs.v[4 * t + 2 * i + 1] * 16u + cs.v[4 * t + 2 * i];
            const uint32_t r = age_nibbles(u, a[2 * i + 1] * 16u + a[2 * i], p.last, p.two);
            a[2 * i] = r & 0x0F0F0F0Fu;
            a[2 * i + 1] = (r >> 4) & 0x0F0F0F0Fu;
          }
        }
        if (!odd_out || to[t].cells == 16) *reinterpret_cast<uint4 *>(q) = make_uint4(a[0], a[1], a[2], a[3]);
        else store_part(q, a, to[t].cells);
      }
    }
  };

  // EDGE: a strip at the top or bottom of the grid, whose rows outside it are
  // zero (the loads stay on rows that exist)
  auto walk = [&](auto edge) {
    constexpr bool EDGE = decltype(edge)::value;
    auto valid_of = [&](int i) { return EDGE && (i < lo || i >= hi) ? 0u : mask; };
    auto load = [&](Raw<SI> &r, int i) {   // row i of the strip's rows
#pragma unroll
      for (int t = 0; t < kParts; ++t) {
        const int row = !EDGE ? i : i < from[t].lo ? from[t].lo : i >= from[t].hi ? from[t].hi - 1 : i;
        const uint8_t *q = row_ptr(from[t].base, (uint32_t)row, pitch);
        if constexpr (SI == CAT_STORE_BIT1) r.v[0] = *reinterpret_cast<const uint32_t *>(q);
        else ld16(r.v + 4 * t, q);
      }
    };
    Raw<SI> raw[A], ctr[2];
#pragma unroll
    for (int k = 0; k < A; ++k) load(raw[k], k);
    if constexpr (MS) {   // centre rows, for their states
      load(ctr[0], R);
      load(ctr[1], R + 1);
    }
    uint32_t S[NS];
#pragma unroll
    for (int b = 0; b < NS; ++b) S[b] = 0u;
    int slot = 0, cslot = 0;

    // Rows go in pairs, whose chains of dependent operations overlap.
    auto take = [&](int i, int k) {   // flags of row i from raw[k], which then takes row i + A
      const uint32_t c = flags_of(raw[k], valid_of(i));
      load(raw[k], i + A);
      return c;
    };
    auto first_rows = [&](int i, int k) {   // rows i, i + 1 < 2 R: into the sum only
      uint32_t h0[NH], h1[NH];
      const uint32_t c0 = take(i, k), c1 = take(i + 1, k + 1);
      hsum(c0, h0);
      hsum(c1, h1);
      ring_store<NH, NT>(smem + next_slot(slot), lane, h0);
      ring_store<NH, NT>(smem + next_slot(slot), lane, h1);
      *reinterpret_cast<uint32_t *>(cring + next_cslot(cslot) + 4 * lane) = c0;
      *reinterpret_cast<uint32_t *>(cring + next_cslot(cslot) + 4 * lane) = c1;
      add_rows(S, h0);
      add_rows(S, h1);
    };
    constexpr int kRest = (2 * R) % A;
    for (int i = 0; i < 2 * R - kRest; i += A) {
#pragma unroll
      for (int k = 0; k < A; k += 2) first_rows(i + k, k);
    }
#pragma unroll
    for (int k = 0; k < kRest; k += 2) first_rows(2 * R - kRest + k, k);
    {   // no row leaves the window of the first output row
      uint32_t z[NH];
#pragma unroll
      for (int b = 0; b < NH; ++b) z[b] = 0u;
      ring_store<NH, NT>(smem + slot, lane, z);
    }

    for (int j = 0; j < p.rows; j += A) {
#pragma unroll
      for (int k = 0; k < A; k += 2) {
        constexpr int kOdd = kRest;
        uint32_t h0[NH], h1[NH], o0[NH], o1[NH], m0, m1;
        const int i = 2 * R + j + k;
        const uint32_t c0 = take(i, (k + kOdd) % A), c1 = take(i + 1, (k + 1 + kOdd) % A);
        hsum(c0, h0);
        hsum(c1, h1);
        uint8_t *const s0 = smem + next_slot(slot), *const s1 = smem + next_slot(slot);
        ring_load<NH, NT>(s0, lane, o0);
        ring_load<NH, NT>(s1, lane, o1);
        ring_store<NH, NT>(s0, lane, h0);
        ring_store<NH, NT>(s1, lane, h1);
        uint32_t *const q0 = reinterpret_cast<uint32_t *>(cring + next_cslot(cslot) + 4 * lane);
        uint32_t *const q1 = reinterpret_cast<uint32_t *>(cring + next_cslot(cslot) + 4 * lane);
        m0 = *q0;
        *q0 = c0;
        m1 = *q1;   // (the same word as q0 when R = 1)
        *q1 = c1;
        if (MS && odd_in) {
          clear_past(ctr[0]);
          clear_past(ctr[1]);
        }
        slide(S, h0, o0);
        const uint32_t in0 = rule(S, m0);
        slide(S, h1, o1);
        const uint32_t in1 = rule(S, m1);
        put(j + k, in0, ctr[0]);
        put(j + k + 1, in1, ctr[1]);
        if constexpr (MS) {
          load(ctr[0], R + j + k + 2);
          load(ctr[1], R + j + k + 3);
        }
      }
    }
  };
  if (inside) walk(std::false_type{});
  else walk(std::true_type{});
}

template <int R, int SI, int SO, bool MS>
__global__ void __launch_bounds__(32, Cfg<R, MS>::kWarps) planes_kernel(const __grid_constant__ Params p) {
  extern __shared__ __align__(16) uint8_t smem[];
  planes_step<R, SI, SO, MS>(p, (int)blockIdx.x, smem);
}

// Batches of two-state uint8 grids, several steps per call on states kept one
// bit per cell, within the rows of whichever of a grid's buffers holds no
// state that is still needed (as one grid's steps are): the bytes are packed,
// stepped and unpacked by separate launches, since the small grids' few warps
// do not keep enough bytes in flight to step from them (512 uneven grids, 4
// steps: 465 us with the first and last step on bytes, 371 us so; the tiles, which
// serve so short calls, 351).
struct BatchGrid {
  uint8_t *buf[2];
  int64_t pitch;
  int32_t H, W, seg, rows, strips;
  int32_t r;
  int32_t cur;       // the buffer that holds the states when the table is made
  int32_t second;    // byte offset of a row's second row of bits
  uint32_t bound[4][kMaxS];
};
struct BatchBlock {   // what a warp (a block when packing) does; grid < 0: nothing
  int32_t grid, block;
};
struct BatchParams {
  const BatchGrid *grids;
  const BatchBlock *blocks;
  int32_t flip;          // steps since the table was made, mod 2
  int32_t step, steps;   // this launch's step of the call's
};

// Where the packed states after t steps of a call lie: in the buffer that does
// not take the final states, but for the first ones (t = 0), which must leave
// the buffer that they are packed from.  (Table reads: nothing writes a table
// while a launch may read it.)
__device__ __forceinline__ uint8_t *packed_place(const BatchGrid *g, int cur, int t, int steps) {
  const bool odd = steps & 1;
  const int b = t == 0 || !odd ? 1 - cur : cur;
  const bool second = odd ? t > 0 && !(t & 1) : t & 1;
  return reinterpret_cast<uint8_t *>(__ldg(reinterpret_cast<const unsigned long long *>(&g->buf[b]))) +
         (second ? __ldg(&g->second) : 0);
}

template <int R>
__device__ __forceinline__ void batch_step(const BatchParams &b, const BatchGrid *g, int block) {
  extern __shared__ __align__(16) uint8_t smem[];
  const int cur = __ldg(&g->cur) ^ b.flip;
  Params p;
  p.in = packed_place(g, cur, b.step, b.steps);
  p.out = packed_place(g, cur, b.step + 1, b.steps);
  p.pitch = __ldg(reinterpret_cast<const long long *>(&g->pitch));
  p.H = __ldg(&g->H);
  p.W = __ldg(&g->W);
  // the last step's row goes on to the end of its last 16 cells, like the
  // tensor-core kernels' stores, which cover whole 16-byte units: the bytes there
  // are the same on both routes of a batch (the first step's input ends at W)
  p.written = b.step == b.steps - 1 ? (p.W + 15) & ~15 : p.W;
  p.seg = __ldg(&g->seg);
  p.rows = __ldg(&g->rows);
  p.strips = __ldg(&g->strips);
  p.frame = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int i = 0; i < Dim<R>::kS; ++i) p.bound[k][i] = __ldg(&g->bound[k][i]);
  planes_step<R, CAT_STORE_BIT1, CAT_STORE_BIT1, false, 2>(p, block, smem + (threadIdx.x >> 5) * Cfg<R, false>::kSmem);
}

// One launch serves the radii LO .. HI, and the warps of a block serve one
// radius: an SM then runs the code of one or two radii at a time.  (Radii mixed
// warp by warp, or sixteen launches side by side, fetch more code than the
// instruction caches hold: 128 grids of 1024^2, 4 steps, one radius 224 us,
// eight radii 777 us; for the same reason the loop is unrolled by two rows.)
constexpr int kBatchWarps = 8;
template <int LO, int HI, int R = LO>
__device__ __forceinline__ void batch_pick(const BatchParams &b, const BatchGrid *g, int block) {
  if constexpr (R <= HI) {
    if (__ldg(&g->r) == R) batch_step<R>(b, g, block);
    else batch_pick<LO, HI, R + 1>(b, g, block);
  }
}
template <int LO, int HI>
__global__ void __launch_bounds__(32 * kBatchWarps, (Cfg<HI, false>::kWarps + kBatchWarps - 1) / kBatchWarps)
    planes_batch_kernel(const __grid_constant__ BatchParams b) {
  const int2 at = __ldg(reinterpret_cast<const int2 *>(b.blocks) + blockIdx.x * kBatchWarps + (threadIdx.x >> 5));
  if (at.x < 0) return;
  batch_pick<LO, HI>(b, b.grids + at.x, at.y);
}

// Kernel of radius r for one storage, with the bytes of shared memory a warp
// takes; nullptr when it is not built.
struct Kernel {
  void (*fn)(Params) = nullptr;
  int smem = 0, ahead = 0, planes = 0;
};
// r <= kMaxR; uint8 with two states and with 3 .. 16, from uint8 to one bit per
// cell and back
Kernel kernel_u8(int r);
Kernel kernel_u8_ms(int r);
Kernel kernel_u8_to_bit1(int r);
Kernel kernel_bit1_to_u8(int r);
Kernel kernel_bit1(int r);
Kernel kernel_nib4(int r);

template <int SI, int SO, bool MS, int LO = 1>
Kernel find_kernel(int r) {
  if constexpr (LO > kMaxR) {
    return Kernel{};
  } else {
    if (r == LO) return Kernel{planes_kernel<LO, SI, SO, MS>, Cfg<LO, MS>::kSmem, Cfg<LO, MS>::kAhead, Dim<LO>::kS};
    return find_kernel<SI, SO, MS, LO + 1>(r);
  }
}

// The batch kernels: of three ranges of radii (a launch's blocks take the shared
// memory of its largest radius), and from bytes (step 0 of the parameters) and
// back (step = steps).
constexpr int kRanges = 3, kRangeEnd[kRanges] = {7, 11, kMaxR};
constexpr int kPackWords = 2048, kPackThreads = 256;   // words per block, threads
typedef void (*BatchFn)(BatchParams);
BatchFn batch_kernel(int range);
BatchFn batch_pack_kernel(bool unpack);

}  // namespace planes
}  // namespace cat
