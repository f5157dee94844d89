// eval_slice.cuh -- the bit-sliced population evaluator (Algorithm 1, Section
// 3.2): device code shared by its translation units.
//
// Samples are processed as bits of 32-bit words.  A tile is 1024 samples: 32
// words, one row of 128 bytes.  A tile's ranks are transposed into bit planes
// (row b of a feature: bit b of every sample's rank) and its labels into one
// row per class -- by planes_kernel (eval_slice.cu) once for the generations of
// a fit, or by the evaluator itself for one evaluation.  The evaluator expands
// the planes of a feature in shared memory into thermometer rows: the rank is
// cut into ND digits of w_j bits, and row T_j[v] holds "digit j >= v" of every
// sample.  "rank >= theta" of 1024 samples is then
//   g = T_low[v_low];   g = T_j[v_j + 1] | (T_j[v_j] & g)   for the higher digits
// -- 2 ND - 1 row loads and one 3-input logic operation per higher digit and
// word, whatever the samples.  All 2^D - 1 nodes of a tree are evaluated this
// way (no divergence, no ballots), the leaf masks are their conjunctions, and a
// bin's count is the population count of leaf AND class.
//
// A warp works on four trees at once: eight lanes each, a lane holding four of
// the 32 words, so that every row load is one 16-byte load per lane and each
// quarter warp reads one whole row (128 bytes: no bank conflicts, whichever
// rows the four trees need).
//
// Bound: shared-memory row loads (4 (2 ND - 1) + record wavefronts per node and four
// trees) with the population counts next (32 per eight leaves, class present and
// four trees, at a quarter of the warp rate or less).  Planes in memory hold a
// fit's samples ordered by class, so that all but K - 1 tiles have one class and
// need no class masks and one count per leaf, whatever K.  One CTA of 16 warps per
// SM: the thermometer rows fill shared memory (12 warps equal, 20 to 32 warps 13 to
// 34% slower: fewer registers than the masks of eight leaves need).
//
// Measured on GB300, per launch (before: the re-laid kernel, whose warps route 32
// samples by ballots, 34 instructions per 32 evaluations against 6.2 here): n = 1e7,
// F = 10, K = 2, 1024 trees of depth 4, uint16: 10.2 ms -> 3.6 ms; n = 1e6, F = 30,
// K = 4, 128 trees of depth 3, uint32: 142 -> 86 us; depth 2: 107 -> 55 us; n = 6e4,
// F = 24, K = 5, 128 trees of depth 3: 23.0 -> 12.6 us; n = 2e6, 256 trees of depth
// 5: 779 -> 390 us.  Depth 6 would be 298 (shared atomics) -> 620 us: every node is
// evaluated for every sample, so the work doubles with each level.
#pragma once

#include "eval_kernel.cuh"

namespace deoct {
namespace slc {

constexpr int kTile = 1024;      // samples per tile (32 words of 32)
constexpr int kWarps = 16;       // warps per CTA (128 registers a thread)
constexpr int kTreesPerWarp = 4;
constexpr int kMaxDigits = 12;
constexpr int kMaxWidth = 6;     // widest digit: 64 rows
constexpr int kFlushTiles = 63;  // tiles a 16-bit bin count holds (63 x 1024 < 2^16)
constexpr int kMaxDepthSlice = 5;
constexpr uint32_t kTheta16 = 65536u;  // uint16 ranks: every larger theta sends all samples left, as this one

struct SliceArgs {
  evk::EvalArgs e;  // S = kTile; tmap, lab_stage and nstage unused
  int rows;         // thermometer rows in shared memory
  int ymask_off, rec_off, acc_off, smem_bytes;
  int rec_bytes;    // node records of one warp
};

// Digit counts the kernel is built for, ascending.
__host__ __device__ constexpr int digit_step(int nd) { return nd < 8 ? nd + 1 : nd + 2; }

// Thermometer rows of one feature cut into nd digits (the widths differ by at
// most one, the wider ones last), 0 when a digit would be wider than kMaxWidth.
__host__ __device__ __forceinline__ int digit_rows(int bits, int nd) {
  const int w = bits / nd, e = bits - w * nd;
  if (w + (e ? 1 : 0) > kMaxWidth || w < 1) return 0;
  return (nd - e) * (1 << w) + e * (2 << w);
}
// Rows of a tile in memory: planes, one row per class, one of any class, and one
// whose first word holds the classes present (class_rows).
__host__ __device__ __forceinline__ int slice_rows(int F, int K, int nb) { return F * nb + K + 2; }
// The fewest digits whose rows fit `rows` for F features (0: none).  One more
// row follows the last feature (see the row layout at Digits).
__host__ __device__ __forceinline__ int pick_digits(int bits, int F, int rows) {
  for (int nd = 1; nd <= kMaxDigits && nd <= bits; nd = digit_step(nd)) {
    const int r = digit_rows(bits, nd);
    if (r > 0 && r * F + 1 <= rows) return nd;
  }
  return 0;
}

// A tree is worked on in subtrees of at most eight leaves, whose counts of one
// class are kept as 16-bit pairs: kWords words.
template <int D>
struct Shape {
  static constexpr int kSubDepth = D < 3 ? D : 3;
  static constexpr int kPrefix = D - kSubDepth;       // levels above the subtrees
  static constexpr int kSubs = 1 << kPrefix;
  static constexpr int kLeaves = 1 << kSubDepth;      // leaves of a subtree
  static constexpr int kWords = kLeaves / 2;
};
// words of a tree's counts: [subtree][class][leaf pair]
__host__ __device__ __forceinline__ int count_words(int D, int K) { return (1 << D) / 2 * K; }

// Bytes from one tree's records to the next tree's, for a subtree's nodes and for
// the prefix nodes: odd multiples of 16, so that the four trees' records lie in
// different banks.  rb: bytes of a record.
__host__ __device__ constexpr int rec_stride(int rb) { return 8 * rb + 16; }
__host__ __device__ constexpr int prefix_stride(int D, int rb) {
  return D > 3 ? ((((1 << (D - 3)) - 1) * rb / 16) | 1) * 16 : 0;
}
__host__ __device__ constexpr int warp_rec_bytes(int D, int rb) {
  return kTreesPerWarp * (rec_stride(rb) + prefix_stride(D, rb));
}

// How a feature's rank is cut into digits (digit 0 is the most significant).
// Rows of a feature, `stride` of them from its base: digit 0 runs upward from a
// row of ones (T[0]) to T[2^w - 1], digit 1 downward from a row of zeros
// (T[2^w] of both digits) to T[1], digit 2 upward from a row of ones again
// (T[0] of both), and so on: neighbours share their constant rows, and T[v + 1]
// is the row after T[v] in an even digit, before it in an odd one.
struct Digits {
  int bits, stride;
  int base[kMaxDigits];   // first (constant) row of the digit
  int shift[kMaxDigits];  // its lowest bit
  int width[kMaxDigits];
  int4 rec[kMaxDigits];   // shift, mask and byte offset of the row of value 0 from the feature's first
  uint32_t bit_row[24];   // row where stage_raw leaves the plane of a bit
};
// Thread j < nd sets digit j: nd - e digits of w bits, then e of w + 1.
__device__ __forceinline__ void set_digits(Digits* d, int bits, int nd) {
  const int w = bits / nd, e = bits - w * nd, n0 = nd - e;
  const int j = threadIdx.x;
  if (j < nd) {
    const int wj = w + (j >= n0 ? 1 : 0);
    const int row = j <= n0 ? j << w : (n0 << w) + ((j - n0) << (w + 1));
    const int top = j <= n0 ? bits - j * w : bits - n0 * w - (j - n0) * (w + 1);  // bits from this digit down
    const int sh = top - wj;
    d->base[j] = row;
    d->shift[j] = sh;
    d->width[j] = wj;
    d->rec[j] = make_int4(sh, (1 << wj) - 1, (row + ((j & 1) ? 1 << wj : 0)) * 128, 0);
    for (int i = 0; i < wj; ++i) d->bit_row[sh + i] = (uint32_t)(row + 1 + i);
  }
  if (j == 0) {
    d->bits = bits;
    d->stride = (n0 << w) + (e << (w + 1));
  }
}

__device__ __forceinline__ uint4 lds4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts1(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v));
}
__device__ __forceinline__ void sts4(uint32_t a, const uint4& v) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w));
}
// Four words of global memory (read-only during the launch) if `on`, else 0.
// Volatile, so that a run of them stays together ahead of the stores that follow.
__device__ __forceinline__ uint4 ldg4_if(const uint32_t* p, bool on) {
  uint4 v;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %5, 0;\n\tmov.u32 %0, 0;\n\tmov.u32 %1, 0;\n\tmov.u32 %2, 0;\n\t"
      "mov.u32 %3, 0;\n\t@q ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p), "r"((int)on));
  return v;
}
__device__ __forceinline__ uint4 and4(const uint4& a, const uint4& b) {
  return make_uint4(a.x & b.x, a.y & b.y, a.z & b.z, a.w & b.w);
}
__device__ __forceinline__ uint4 andn4(const uint4& a, const uint4& b) {
  return make_uint4(a.x & ~b.x, a.y & ~b.y, a.z & ~b.z, a.w & ~b.w);
}
__device__ __forceinline__ uint4 or4(const uint4& a, const uint4& b) {
  return make_uint4(a.x | b.x, a.y | b.y, a.z | b.z, a.w | b.w);
}

// ---------------------------------------------------------------------------
// thermometer rows
// ---------------------------------------------------------------------------
// The rows T[v], v = 1 .. 2^W - 1 ("digit >= v"), of a digit from its planes b,
// most significant bit first: with x standing for the comparison of the bits
// below, T is o | (a & x), and a bit of v that is 0 makes x into b | x, one that is
// 1 into b & x.  Upward digits keep T[v] at row v, downward ones at row 2^W - v.
template <int W, bool UP, int L, int V>
__device__ __forceinline__ void emit_rows(const uint4* b, const uint4& o, const uint4& a, uint32_t sa) {
  constexpr int r0 = UP ? V : (1 << W) - V, r1 = UP ? V + 1 : (1 << W) - V - 1;
  if constexpr (L == 1) {
    if constexpr (V > 0) sts4(sa + r0 * 128, or4(o, a));
    sts4(sa + r1 * 128, or4(o, and4(a, b[0])));
  } else {
    const uint4 ab = and4(a, b[L - 1]);
    emit_rows<W, UP, L - 1, V>(b, or4(o, ab), a, sa);
    emit_rows<W, UP, L - 1, V + (1 << (L - 1))>(b, o, ab, sa);
  }
}
template <int W, bool UP>
__device__ __forceinline__ void store_digit(const uint4* b, uint32_t sa) {
  emit_rows<W, UP, W, 0>(b, make_uint4(0u, 0u, 0u, 0u), make_uint4(~0u, ~0u, ~0u, ~0u), sa);
}

// Widest digit a count of ND digits meets (ranks of at most 24 bits).
template <int ND>
struct MaxWidth {
  static constexpr int k = (24 + ND - 1) / ND < kMaxWidth ? (24 + ND - 1) / ND : kMaxWidth;
};

// 16 x 16 bit transposes of the low and of the high halves of x[0..15]:
// afterwards bit i (16 + i) of x[b] is bit b of the low (high) half of the old x[i].
template <int S>
__device__ __forceinline__ void transpose_stage(uint32_t (&x)[16]) {
  constexpr uint32_t m = S == 8 ? 0x00FF00FFu : S == 4 ? 0x0F0F0F0Fu : S == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
  for (int p = 0; p < 8; ++p) {  // the pairs (k, k + S): bit S of k is clear
    const int k = (p / S) * 2 * S + p % S;
    const uint32_t t = ((x[k] >> S) ^ x[k + S]) & m;
    x[k + S] ^= t;
    x[k] ^= t << S;
  }
}
__device__ __forceinline__ void transpose16(uint32_t (&x)[16]) {
  transpose_stage<8>(x);
  transpose_stage<4>(x);
  transpose_stage<2>(x);
  transpose_stage<1>(x);
}

// Samples s0 .. s0 + ns of a problem's segment.
struct TileSpan {
  int64_t s0;
  int ns;
};
__device__ __forceinline__ TileSpan tile_span(const EvalProb& P, int64_t tile) {
  TileSpan t;
  const int64_t j0 = tile * kTile;
  t.s0 = P.start + j0;
  t.ns = P.count - j0 < kTile ? (int)(P.count - j0) : kTile;
  return t;
}
__device__ __forceinline__ int64_t column_of(const EvalProb& P, int64_t s, int* status) {
  if (!P.idx) return s;
  const int64_t col = P.idx[s];
  if ((uint64_t)col < (uint64_t)P.ncols) return col;
  atomicOr(status, ST_BAD_INDEX);
  return 0;
}

// The lane's 32 samples of one feature of a tile: v[i] holds samples 64 i + 2 lane
// and the next (uint16: as one word; uint32: two), 0 past the end.  They become
// bits i and 16 + i of word `lane`, so a warp's loads are coalesced.
template <int W>
struct RawWords {
  uint32_t lo[16], hi[W == 4 ? 16 : 1];
};
template <int W>
__device__ __forceinline__ void load_raw(const EvalProb& P, const TileSpan& t, int f, int lane, int* status,
                                         RawWords<W>& v) {
  typedef typename evk::RankT<W>::T RT;
  const RT* row = static_cast<const RT*>(P.ranks) + (int64_t)f * P.ld;
  if (P.tma && t.ns == kTile) {
    const char* r = reinterpret_cast<const char*>(row + t.s0) + lane * 2 * W;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if constexpr (W == 2)
        asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(v.lo[i]) : "l"(r + i * 128));
      else
        asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.lo[i]), "=r"(v.hi[i]) : "l"(r + i * 256));
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int j = 64 * i + 2 * lane;
    const uint32_t a = j < t.ns ? (uint32_t)row[column_of(P, t.s0 + j, status)] : 0u;
    const uint32_t b = j + 1 < t.ns ? (uint32_t)row[column_of(P, t.s0 + j + 1, status)] : 0u;
    if constexpr (W == 2) {
      v.lo[i] = a | b << 16;
    } else {
      v.lo[i] = a;
      v.hi[i] = b;
    }
  }
}
// Word `lane` of every bit plane: planes 0..15 in x, 16..23 in h (uint32 ranks).
// Ranks saturate at 2^bits - 1, which no theta exceeds.
template <int W>
__device__ __forceinline__ void raw_planes(const RawWords<W>& v, int bits, uint32_t (&x)[16], uint32_t (&h)[16]) {
  const uint32_t top = (1u << bits) - 1u;  // bits <= 24
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    if constexpr (W == 2) {
      x[i] = bits < 16 ? __vminu2(v.lo[i], top | top << 16) : v.lo[i];
    } else {
      const uint32_t a = min(v.lo[i], top), b = min(v.hi[i], top);
      x[i] = __byte_perm(a, b, 0x5410);
      h[i] = __byte_perm(a, b, 0x7632);
    }
  }
  if constexpr (W == 4) {
    if (bits > 16) transpose16(h);
  }
  transpose16(x);
}

// The labels of the lane's 32 samples as 16-bit pairs (samples 64 i + 2 lane and
// the next; 0xFFFF past the end: in no class), and their class-k word.
__device__ __forceinline__ void label_pairs(const EvalProb& P, const TileSpan& t, int lane, int* status,
                                            uint32_t (&la)[16]) {
  if (P.tma && P.lab_tma && t.ns == kTile) {  // aligned labels, read in pairs
    const char* y = reinterpret_cast<const char*>(P.labels + t.s0) + lane * 2;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      unsigned short v;
      asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(v) : "l"(y + i * 64));
      la[i] = __byte_perm(v, 0u, 0x4140);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const int j = 64 * i + 2 * lane;
    uint32_t y0 = 0xFFFFu, y1 = 0xFFFFu;
    if (j < t.ns) y0 = P.labels[column_of(P, t.s0 + j, status)];
    if (j + 1 < t.ns) y1 = P.labels[column_of(P, t.s0 + j + 1, status)];
    la[i] = y0 | y1 << 16;
  }
}
__device__ __forceinline__ uint32_t class_word(const uint32_t (&la)[16], uint32_t k) {
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    m |= ((la[i] & 0xFFFFu) == k ? 1u : 0u) << i;
    m |= ((la[i] >> 16) == k ? 1u : 0u) << (16 + i);
  }
  return m;
}

// The class rows of a tile, called by one warp: word `lane` of row k and of row K
// (samples of any class), and the least and the largest class present, packed
// (k0 | k1 << 16; k0 = k1 = 0 for a tile without valid labels).
template <typename Put>
__device__ __forceinline__ uint32_t class_rows(const EvalProb& P, const TileSpan& t, int lane, int* status, Put put) {
  uint32_t la[16];
  label_pairs(P, t, lane, status, la);
  uint32_t any = 0, k0 = 0xFFFFu, k1 = 0;
  for (int k = 0; k < P.K; ++k) {
    const uint32_t y = class_word(la, (uint32_t)k);
    if (__any_sync(0xFFFFFFFFu, y != 0u)) {
      k0 = min(k0, (uint32_t)k);
      k1 = (uint32_t)k;
    }
    any |= y;
    put(k, y);
  }
  put(P.K, any);
  return k0 == 0xFFFFu ? 0u : k0 | k1 << 16;
}

// A tile without planes in memory: its ranks transposed here.  The planes of a
// feature wait in its own thermometer rows (digit j's planes in the first rows
// after its constant one).
template <int W>
__device__ __forceinline__ void stage_raw(const Digits* dg, const EvalProb& P, int tile, uint32_t therm_sa,
                                          uint32_t ymask_sa, uint32_t* s_classes, int lane, int warp, int* status) {
  const TileSpan t = tile_span(P, tile);
  const int bits = dg->bits, stride = dg->stride, F = P.F;
  constexpr int kStagers = kWarps - 1;  // the last warp has the class rows
  if (warp == kStagers) {
    const uint32_t c = class_rows(P, t, lane, status, [&](int k, uint32_t y) { sts1(ymask_sa + k * 128 + lane * 4, y); });
    if (lane == 0) *s_classes = c;
    return;
  }
  for (int f = warp; f < F; f += kStagers) {
    RawWords<W> v;
    load_raw<W>(P, t, f, lane, status, v);
    uint32_t x[16], h[16];
    raw_planes<W>(v, bits, x, h);
    const uint32_t fsa = therm_sa + (uint32_t)(f * stride) * 128u + (uint32_t)lane * 4u;
#pragma unroll
    for (int b = 0; b < 16; ++b)
      if (b < bits) sts1(fsa + dg->bit_row[b] * 128u, x[b]);
    if constexpr (W == 4) {
#pragma unroll
      for (int b = 0; b < 8; ++b)
        if (16 + b < bits) sts1(fsa + dg->bit_row[16 + b] * 128u, h[b]);
    } else if (bits > 16) {
      sts1(fsa + dg->bit_row[16] * 128u, 0u);
    }
  }
}

// Expand a tile's planes into thermometer rows and copy its class rows, all
// warps together.  A task is one digit of four features, eight lanes and four
// words a lane each (16-byte loads and stores; a warp per feature with one word a
// lane took three times as long); a task's planes are loaded while the one before
// it is expanded.  blk: the tile's planes, or nullptr when stage_raw left them here.
template <int ND, bool RAW>
__device__ __forceinline__ void build_tile(const Digits* dg, const uint32_t* blk, int F, int K, int nb,
                                           uint32_t therm_sa, uint32_t ymask_sa, uint32_t* s_classes, int lane,
                                           int warp) {
  constexpr int MW = MaxWidth<ND>::k;
  const int q = lane >> 3, l8 = lane & 7;
  const uint32_t fstep = (uint32_t)dg->stride * 128u;
  const int ntask = ((F + 3) >> 2) * ND;
  auto load = [&](int task, uint4 (&pl)[MW]) {
    const int g = task / ND, j = task - g * ND, f = 4 * g + q;
    const int w = dg->width[j];
    if constexpr (!RAW) {
      const int sh = dg->shift[j];
      const uint32_t* pf = blk + ((size_t)f * nb + sh) * 32 + l8 * 4;
      const int have = f < F ? min(w, nb - sh) : 0;  // planes past the problem's own are zero
#pragma unroll
      for (int i = 0; i < MW; ++i) pl[i] = ldg4_if(pf + i * 32, i < have);
    } else {
      const uint32_t sa = therm_sa + (f < F ? (uint32_t)f * fstep : 0u) + (uint32_t)(dg->base[j] + 1) * 128u + l8 * 16;
#pragma unroll
      for (int i = 0; i < MW; ++i) pl[i] = i < w ? lds4(sa + i * 128) : make_uint4(0, 0, 0, 0);
    }
  };
  constexpr bool kAhead = MW <= 4;  // (wide digits: few tasks a warp, and no registers for two)
  uint4 cur[MW], nxt[kAhead ? MW : 1];
  if (kAhead && warp < ntask) load(warp, cur);
  if (!RAW && warp == kWarps - 1) {  // class rows: four at a time, then the classes present
    const uint32_t* y = blk + (size_t)F * nb * 32;
    for (int k = q; k < K + 1; k += 4) sts4(ymask_sa + k * 128 + l8 * 16, ldg4_if(y + k * 32 + l8 * 4, true));
    if (lane == 0) *s_classes = y[(K + 1) * 32];
  }
  for (int task = warp; task < ntask; task += kWarps) {
    if constexpr (kAhead) {
      if (task + kWarps < ntask) load(task + kWarps, nxt);
    } else {
      load(task, cur);
    }
    const int g = task / ND, j = task - g * ND, f = 4 * g + q;
    if (f < F) {
      const uint32_t sa = therm_sa + (uint32_t)f * fstep + (uint32_t)dg->base[j] * 128u + (uint32_t)l8 * 16u;
      auto put = [&](auto up) {
        constexpr bool UP = decltype(up)::value;
        switch (dg->width[j]) {
          case 1: store_digit<1, UP>(cur, sa); break;
          case 2: if constexpr (MW >= 2) store_digit<2, UP>(cur, sa); break;
          case 3: if constexpr (MW >= 3) store_digit<3, UP>(cur, sa); break;
          case 4: if constexpr (MW >= 4) store_digit<4, UP>(cur, sa); break;
          case 5: if constexpr (MW >= 5) store_digit<5, UP>(cur, sa); break;
          default: if constexpr (MW >= 6) store_digit<6, UP>(cur, sa); break;
        }
      };
      if ((j & 1) == 0) put(std::true_type{});
      else put(std::false_type{});
    }
    if constexpr (kAhead) {
#pragma unroll
      for (int i = 0; i < MW; ++i) cur[i] = nxt[i];
    }
  }
}

// The constant rows of every feature (they hold for all tiles of a job).
template <int ND>
__device__ __forceinline__ void fill_const_rows(const Digits* dg, int F, uint32_t therm_sa) {
  for (int e = threadIdx.x; e < (F * ND + 1) * 8; e += blockDim.x) {
    const int r = e >> 3, f = r / ND, j = r - f * ND;
    // (the row after the last feature, j = 0, closes its last digit)
    const int row = f * dg->stride + (f < F ? dg->base[j] : 0);
    const uint32_t v = (j & 1) ? 0u : 0xFFFFFFFFu;
    sts4(therm_sa + (uint32_t)row * 128u + (uint32_t)(e & 7) * 16u, make_uint4(v, v, v, v));
  }
}

// ---------------------------------------------------------------------------
// nodes
// ---------------------------------------------------------------------------
// A node as feature << 24 | theta.  Trees as given by the caller are validated
// here (a > F, or a theta past the packed range, is flagged and evaluated as a
// no-split node).
struct Trees {
  const uint32_t* nodes;
  const uint16_t* a16;  // nullable: the trees as given, with th32
  const uint32_t* th32;
  int F;
  __device__ __forceinline__ explicit Trees(const EvalProb& P) : nodes(P.nodes), a16(P.a16), th32(P.th32), F(P.F) {}
};
__device__ __forceinline__ uint32_t fetch_node(const Trees& T, int64_t e, int* status) {
  if (T.a16 == nullptr) return T.nodes[e];
  int av = T.a16[e];
  const uint32_t tv = T.th32[e];
  if (av > T.F || (av > 0 && tv > kThetaMask)) {
    atomicOr(status, ST_BAD_NODE);
    av = 0;
  }
  return pack_node(av, tv);
}

// Node record: the shared addresses of T_j[v_j] of every digit.
template <int ND>
struct RecBytes {
  static constexpr int k = (ND + 3) / 4 * 16;
};

// The digits as the records need them: digit j of a threshold is at first[j]
// (byte offset of the row of v = 0 from the feature's first row), and its rows
// run up or down from there.  Held in registers for few digits, else read again
// from shared memory for every record.
template <int ND>
struct RecDigits {
  static constexpr bool kHeld = ND <= 4;
  const Digits* dg;
  int stride;
  int shift[kHeld ? ND : 1], mask[kHeld ? ND : 1], first[kHeld ? ND : 1];
  __device__ __forceinline__ explicit RecDigits(const Digits* d) : dg(d), stride(d->stride * 128) {
    if constexpr (kHeld) {
#pragma unroll
      for (int j = 0; j < ND; ++j) {
        shift[j] = d->rec[j].x;
        mask[j] = d->rec[j].y;
        first[j] = d->rec[j].z;
      }
    }
  }
};

template <int ND>
__device__ __forceinline__ void put_record(const RecDigits<ND>& rd, uint32_t node, uint32_t tmax, uint32_t therm_sa,
                                           unsigned char* rec) {
  const uint32_t f = node >> 24;
  uint32_t th = node & kThetaMask;
  th = th > tmax ? tmax : th;
  const uint32_t fr = therm_sa + f * (uint32_t)rd.stride;
  uint32_t a[RecBytes<ND>::k / 4];
#pragma unroll
  for (int j = 0; j < RecBytes<ND>::k / 4; ++j) {
    if (j >= ND) {
      a[j] = 0u;
      continue;
    }
    int shift, mask, first;
    if constexpr (RecDigits<ND>::kHeld) {
      shift = rd.shift[j];
      mask = rd.mask[j];
      first = rd.first[j];
    } else {
      const int4 c = rd.dg->rec[j];
      shift = c.x;
      mask = c.y;
      first = c.z;
    }
    const uint32_t v = (th >> shift) & (uint32_t)mask;
    a[j] = fr + (uint32_t)first + ((j & 1) ? 0u - v * 128u : v * 128u);
  }
#pragma unroll
  for (int j = 0; j < RecBytes<ND>::k / 16; ++j)
    reinterpret_cast<uint4*>(rec)[j] = make_uint4(a[4 * j], a[4 * j + 1], a[4 * j + 2], a[4 * j + 3]);
}

// "rank >= theta" of the lane's 128 samples; lane_sa: byte offset of the lane's
// words in a row.
template <int ND>
__device__ __forceinline__ uint4 node_mask(uint32_t rec_sa, uint32_t lane_sa) {
  uint32_t a[RecBytes<ND>::k / 4];
#pragma unroll
  for (int j = 0; j < RecBytes<ND>::k / 16; ++j) {
    const uint4 r = lds4(rec_sa + 16 * j);
    a[4 * j] = r.x + lane_sa;
    a[4 * j + 1] = r.y + lane_sa;
    a[4 * j + 2] = r.z + lane_sa;
    a[4 * j + 3] = r.w + lane_sa;
  }
  uint4 g = lds4(a[ND - 1]);
#pragma unroll
  for (int j = ND - 2; j >= 0; --j) {
    const uint4 t = lds4(a[j]);
    const uint4 u = lds4((j & 1) ? a[j] - 128u : a[j] + 128u);
    g.x = u.x | (t.x & g.x);
    g.y = u.y | (t.y & g.y);
    g.z = u.z | (t.z & g.z);
    g.w = u.w | (t.w & g.w);
  }
  return g;
}

// The leaf masks, in leaf order, of a subtree of depth SD whose root is reached by
// the samples of pm: node I of level L splits mask I of its level into masks 2 I
// and 2 I + 1 of the next, from the last node down so that no mask is overwritten
// before it is split.
template <int ND, int SD, int L, int I>
__device__ __forceinline__ void split_masks(uint32_t rec_sa, uint32_t lane_sa, uint4 (&m)[1 << SD]) {
  const uint4 g = node_mask<ND>(rec_sa + (uint32_t)((1 << L) - 1 + I) * RecBytes<ND>::k, lane_sa);
  const uint4 p = m[I];
  m[2 * I + 1] = and4(p, g);
  m[2 * I] = andn4(p, g);
  if constexpr (I > 0) split_masks<ND, SD, L, I - 1>(rec_sa, lane_sa, m);
  else if constexpr (L + 1 < SD) split_masks<ND, SD, L + 1, (2 << L) - 1>(rec_sa, lane_sa, m);
}
template <int ND, int SD>
__device__ __forceinline__ void leaf_masks(uint32_t rec_sa, uint32_t lane_sa, const uint4& pm,
                                           uint4 (&m)[1 << SD]) {
  m[0] = pm;
  split_masks<ND, SD, 0, 0>(rec_sa, lane_sa, m);
}

__device__ __forceinline__ uint32_t pop4(const uint4& v) {
  return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
}

// Sum the packed counts of the eight lanes of a tree (at most 1024 a bin) and add
// them to the tree's counts, which only this warp touches.  The exchanges halve
// the words a lane holds while they can: lane l8 ends with word l8 / (8 / NW).
template <int NW>
__device__ __forceinline__ void add_counts(const uint32_t (&p)[NW], uint32_t* a, int l8, bool on) {
  uint32_t v;
  if constexpr (NW == 4) {
    const bool h4 = l8 & 4, h2 = l8 & 2;
    uint32_t k0 = h4 ? p[2] : p[0], k1 = h4 ? p[3] : p[1];
    k0 += __shfl_xor_sync(0xFFFFFFFFu, h4 ? p[0] : p[2], 4);
    k1 += __shfl_xor_sync(0xFFFFFFFFu, h4 ? p[1] : p[3], 4);
    v = (h2 ? k1 : k0) + __shfl_xor_sync(0xFFFFFFFFu, h2 ? k0 : k1, 2);
  } else if constexpr (NW == 2) {
    const bool h4 = l8 & 4;
    v = (h4 ? p[1] : p[0]) + __shfl_xor_sync(0xFFFFFFFFu, h4 ? p[0] : p[1], 4);
    v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
  } else {
    v = p[0] + __shfl_xor_sync(0xFFFFFFFFu, p[0], 4);
    v += __shfl_xor_sync(0xFFFFFFFFu, v, 2);
  }
  v += __shfl_xor_sync(0xFFFFFFFFu, v, 1);
  constexpr int per = 8 / NW;  // lanes that hold the same word
  if (on && (l8 & (per - 1)) == 0) a[l8 / per] += v;
}

// All trees of the job over the tile in shared memory.  A warp takes four trees
// at a time; lane / 8 tells which, lane % 8 which four words of a row.
template <int D, int ND>
__device__ __forceinline__ void route_tile(const Digits* dg, const EvalProb& P, int tree0, int ntrees, int accw,
                                           uint32_t therm_sa, uint32_t ymask_sa, unsigned char* wrec, uint32_t* accb,
                                           uint32_t classes, int* status, int lane, int warp) {
  const int k0 = (int)(classes & 0xFFFFu), k1 = (int)(classes >> 16);
  typedef Shape<D> S;
  constexpr int B = (1 << D) - 1, NL = S::kLeaves, RB = RecBytes<ND>::k;
  constexpr int SN = NL - 1;  // nodes of a subtree
  const int q = lane >> 3, l8 = lane & 7;
  const uint32_t lane_sa = (uint32_t)l8 * 16u;
  const RecDigits<ND> rd(dg);
  unsigned char* rec = wrec + q * rec_stride(RB);  // the tree's subtree records
  unsigned char* prec = wrec + kTreesPerWarp * rec_stride(RB) + q * prefix_stride(D, RB);  // its prefix records
  const uint32_t rec_sa = smem_u32(rec), prec_sa = smem_u32(prec);
  const uint32_t y_sa = ymask_sa + (uint32_t)l8 * 16u;
  // node of lane l8 in a subtree rooted at the 1-based node t: level lv, offset lo
  const int lv = l8 == 0 ? 0 : (l8 < 3 ? 1 : 2), lo = l8 - ((1 << lv) - 1);
  const Trees T(P);
  const int K = P.K;
  const uint32_t tmax = P.W == 2 ? kTheta16 : kThetaMask;
  const int step = kWarps * kTreesPerWarp;
  auto subtree_node = [&](int i, int j) {  // the lane's packed node of subtree j of local tree i
    const int t = ((S::kSubs + j) << lv) + lo;
    const int ic = i < ntrees ? i : ntrees - 1;
    return l8 < SN ? fetch_node(T, (int64_t)(tree0 + ic) * B + t - 1, status) : 0u;
  };
  int i = warp * kTreesPerWarp + q;
  if (warp * kTreesPerWarp >= ntrees) return;
  uint32_t next = subtree_node(i, 0);
  auto prefix_node = [&](int i) {  // the lane's node above the subtrees of local tree i
    const int ic = i < ntrees ? i : ntrees - 1;
    return l8 < S::kSubs - 1 ? fetch_node(T, (int64_t)(tree0 + ic) * B + l8, status) : 0u;
  };
  static_assert(S::kSubs - 1 <= 8, "a lane per prefix node");
  uint32_t pnext = S::kPrefix > 0 ? prefix_node(i) : 0u;
  for (; i - q < ntrees; i += step) {
    if constexpr (S::kPrefix > 0) {
      __syncwarp();
      if (l8 < S::kSubs - 1) put_record<ND>(rd, pnext, tmax, therm_sa, prec + l8 * RB);
      pnext = prefix_node(i + step);
    }
    uint4 G[S::kPrefix > 0 ? S::kPrefix : 1];
    uint32_t* acc = accb + (i < ntrees ? i : 0) * accw;
#pragma unroll 1
    for (int j = 0; j < S::kSubs; ++j) {
      __syncwarp();  // every lane is done with the previous records
      if (l8 < SN) put_record<ND>(rd, next, tmax, therm_sa, rec + l8 * RB);
      __syncwarp();
      // the next subtree's nodes arrive while this one is routed
      if (j + 1 < S::kSubs) next = subtree_node(i, j + 1);
      else if (i - q + step < ntrees) next = subtree_node(i + step, 0);
      uint4 m[NL];
      uint4 pm = lds4(y_sa + (uint32_t)K * 128u);  // samples of any class
      if constexpr (S::kPrefix > 0) {
#pragma unroll
        for (int v = 0; v < S::kPrefix; ++v) {
          // level v's node on the way to subtree j: new when j's lower bits are zero
          if ((j & ((1 << (S::kPrefix - v)) - 1)) == 0)
            G[v] = node_mask<ND>(prec_sa + (uint32_t)((1 << v) - 1 + (j >> (S::kPrefix - v))) * RB, lane_sa);
          const uint32_t x = ((j >> (S::kPrefix - 1 - v)) & 1) ? 0u : ~0u;
          pm.x &= G[v].x ^ x;
          pm.y &= G[v].y ^ x;
          pm.z &= G[v].z ^ x;
          pm.w &= G[v].w ^ x;
        }
      }
      leaf_masks<ND, S::kSubDepth>(rec_sa, lane_sa, pm, m);
      // Counts: the leaves' samples of every class present but the last, whose
      // counts are what remains of the leaves' totals.
      uint32_t rest[S::kWords];
#pragma unroll
      for (int h = 0; h < S::kWords; ++h) rest[h] = pop4(m[2 * h]) + (pop4(m[2 * h + 1]) << 16);
      uint32_t* aj = acc + j * K * S::kWords;
      for (int k = k0; k < k1; ++k) {
        const uint4 y = lds4(y_sa + (uint32_t)k * 128u);
        uint32_t p[S::kWords];
#pragma unroll
        for (int h = 0; h < S::kWords; ++h) {
          p[h] = pop4(and4(m[2 * h], y)) + (pop4(and4(m[2 * h + 1], y)) << 16);
          rest[h] -= p[h];
        }
        add_counts(p, aj + k * S::kWords, l8, i < ntrees);
      }
      add_counts(rest, aj + k1 * S::kWords, l8, i < ntrees);
    }
  }
}

// A job's 16-bit counts into its problem's HBM counts (one atomic per nonzero
// bin), zeroed here for the tiles that follow.
template <int D>
__device__ __forceinline__ void flush_counts(const EvalProb& P, int tree0, int ntrees, int accw, uint32_t* acc) {
  typedef Shape<D> S;
  const int K = P.K, per = K * S::kWords;  // words of a subtree
  uint32_t* dst = P.counts + (int64_t)tree0 * 2 * accw;
  for (int e = threadIdx.x; e < ntrees * accw; e += blockDim.x) {
    const uint32_t v = acc[e];
    if (v == 0) continue;
    acc[e] = 0;
    const int tree = e / accw, x = e - tree * accw;
    const int j = x / per, y = x - j * per, k = y / S::kWords, h = y - k * S::kWords;
    uint32_t* d = dst + (int64_t)tree * 2 * accw + (j * S::kLeaves + 2 * h) * K + k;
    if (v & 0xFFFFu) atomicAdd(d, v & 0xFFFFu);
    if (v >> 16) atomicAdd(d + K, v >> 16);
  }
}

// A tile whose trees hold a theta with more bits than the launch has rows for (the
// launch is sized from the set's size, which bounds the ranks of an encoded set;
// a set that is a view of a larger one, or thetas past n_p, may exceed it): every
// sample walks every tree from global memory.
template <int D>
__device__ __noinline__ void route_general(const EvalProb& P, int tile, int tree0, int ntrees, int* status) {
  constexpr int B = (1 << D) - 1;
  const Trees T(P);
  const TileSpan t = tile_span(P, tile);
  for (int e = threadIdx.x; e < ntrees * kTile; e += blockDim.x) {
    const int i = e / kTile, j = e - i * kTile;
    if (j >= t.ns) continue;
    const int64_t col = column_of(P, t.s0 + j, status);
    int v = 1;
#pragma unroll 1
    for (int d = 0; d < D; ++d) {
      const uint32_t nd = fetch_node(T, (int64_t)(tree0 + i) * B + v - 1, status);
      const int64_t at = (int64_t)(nd >> 24) * P.ld + col;
      const uint32_t rank = P.W == 2 ? static_cast<const uint16_t*>(P.ranks)[at] : static_cast<const uint32_t*>(P.ranks)[at];
      v = 2 * v + (rank >= (nd & kThetaMask) ? 1 : 0);
    }
    const int y = P.labels[col];
    if (y < P.K) atomicAdd(P.counts + ((int64_t)(tree0 + i) * (B + 1) + v - (B + 1)) * P.K + y, 1u);
  }
}

// RAW: no problem of the launch has planes; otherwise all have.
template <int D, int ND, bool RAW>
__global__ void __launch_bounds__(kWarps * 32, 1) eval_slice_kernel(const __grid_constant__ SliceArgs sa) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ Digits dg;
  __shared__ uint32_t s_max;
  __shared__ uint32_t s_classes;  // least and largest class of the tile (class_rows)
  const evk::EvalArgs& a = sa.e;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t therm_sa = smem_u32(smem), ymask_sa = therm_sa + (uint32_t)sa.ymask_off;
  uint32_t* acc = reinterpret_cast<uint32_t*>(smem + sa.acc_off);
  const int64_t T = a.total_tiles;
  const int64_t t0 = (int64_t)blockIdx.x * T / gridDim.x;
  const int64_t t1 = (int64_t)(blockIdx.x + 1) * T / gridDim.x;
  bool fit = true;  // the job's thetas fit the rows (uniform)
  int cur_job = -1, held = 0;  // held: tiles in the 16-bit counts
  evk::JobView jv;
  unsigned char* rec = smem + sa.rec_off + warp * sa.rec_bytes;
  int accw = 0;
  for (int64_t gt = t0; gt < t1; ++gt) {
    evk::JobView nv;
    if (gt == t0) {
      evk::lookup_job(a, gt, &nv);
    } else {
      nv = jv;
      evk::advance_job(a, gt, &nv);
    }
    __syncthreads();  // every warp is done with the previous tile
    if (nv.job != cur_job || held == kFlushTiles) {
      if (cur_job >= 0) flush_counts<D>(*jv.p, jv.tree0, jv.ntrees, accw, acc);
      held = 0;
    }
    if (nv.job != cur_job) {
      __syncthreads();  // the flush reads the digits of no job, but its counts are zeroed below
      const EvalProb& P = *nv.p;
      accw = count_words(D, P.K);
      if (RAW) {  // the planes in use: those of the largest theta of the job's trees
        if (threadIdx.x == 0) s_max = 0;
        __syncthreads();
        const Trees T(P);
        uint32_t mx = 0;
        for (int e = threadIdx.x; e < nv.ntrees * ((1 << D) - 1); e += blockDim.x)
          mx = max(mx, fetch_node(T, (int64_t)nv.tree0 * ((1 << D) - 1) + e, a.status) & kThetaMask);
        mx = __reduce_max_sync(0xFFFFFFFFu, min(mx, P.W == 2 ? kTheta16 : kThetaMask));
        if (lane == 0) atomicMax(&s_max, mx);
        __syncthreads();
      }
      int bits = RAW ? 32 - __clz(s_max) : P.nb;
      bits = bits < ND ? ND : bits;  // (a bit for every digit; planes past the problem's own are zero)
      fit = digit_rows(bits, ND) > 0 && digit_rows(bits, ND) * P.F + 1 <= sa.rows;
      set_digits(&dg, fit ? bits : ND, ND);
      for (int e = threadIdx.x; e < nv.ntrees * accw; e += blockDim.x) acc[e] = 0;
      __syncthreads();
      fill_const_rows<ND>(&dg, P.F, therm_sa);
      cur_job = nv.job;
    }
    jv = nv;
    const EvalProb& P = *jv.p;
    const size_t bw = (size_t)slice_rows(P.F, P.K, P.nb) * 32;  // words of a tile's planes and class rows
    const uint32_t* blk = RAW ? nullptr : P.planes + (size_t)jv.tile * bw;
    if (RAW && !fit) {
      route_general<D>(P, jv.tile, jv.tree0, jv.ntrees, a.status);
      continue;
    }
    if constexpr (RAW) {
      if (P.W == 2) stage_raw<2>(&dg, P, jv.tile, therm_sa, ymask_sa, &s_classes, lane, warp, a.status);
      else stage_raw<4>(&dg, P, jv.tile, therm_sa, ymask_sa, &s_classes, lane, warp, a.status);
      __syncthreads();  // a digit's task reads planes that other warps left
    }
    build_tile<ND, RAW>(&dg, blk, P.F, P.K, P.nb, therm_sa, ymask_sa, &s_classes, lane, warp);
    // the CTA's next tile on its way to L2 while this one is routed
    if (gt + 1 < t1 && jv.tile + 1 < jv.ntiles) {
      if constexpr (!RAW) {
        const char* nx = reinterpret_cast<const char*>(blk + bw);
        for (size_t o = (size_t)threadIdx.x * 128; o < bw * 4; o += (size_t)blockDim.x * 128)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(nx + o));
      } else if (P.tma) {
        const TileSpan t = tile_span(P, jv.tile + 1);
        const int lines = (t.ns * P.W + 127) >> 7;  // 128-byte lines of a row's tile
        for (int e = threadIdx.x; e < P.F * lines; e += blockDim.x) {
          const int f = e / lines, l = e - f * lines;
          asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char*>(P.ranks) +
                                                        ((int64_t)f * P.ld + t.s0) * P.W + l * 128));
        }
        if (threadIdx.x < 8 && threadIdx.x * 128 < t.ns)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(P.labels + t.s0 + threadIdx.x * 128));
      }
    }
    __syncthreads();
    route_tile<D, ND>(&dg, P, jv.tree0, jv.ntrees, accw, therm_sa, ymask_sa, rec, acc, s_classes, a.status,
                      lane, warp);
    ++held;
  }
  __syncthreads();
  if (cur_job >= 0) flush_counts<D>(*jv.p, jv.tree0, jv.ntrees, accw, acc);
  __syncthreads();
  evk::take_ticket<D>(a, smem, (size_t)sa.smem_bytes);
}

// One launch of the kernel of depth D and ND digits (eval_slice_*.cu).
template <int D, int ND>
int launch_slice_t(deoct_ctx* ctx, const SliceArgs& sa, bool raw, int grid, cudaStream_t s) {
  auto* kern = raw ? eval_slice_kernel<D, ND, true> : eval_slice_kernel<D, ND, false>;
  DEOCT_TRY(set_max_dynamic_smem(ctx, kern));
  return launch_on(ctx, "eval_slice_kernel", kern, grid, kWarps * 32, (size_t)sa.smem_bytes, s, sa);
}
template <int D>
int launch_slice_d(deoct_ctx* ctx, int nd, const SliceArgs& sa, bool raw, int grid, cudaStream_t s) {
  switch (nd) {
    case 1: return launch_slice_t<D, 1>(ctx, sa, raw, grid, s);
    case 2: return launch_slice_t<D, 2>(ctx, sa, raw, grid, s);
    case 3: return launch_slice_t<D, 3>(ctx, sa, raw, grid, s);
    case 4: return launch_slice_t<D, 4>(ctx, sa, raw, grid, s);
    case 5: return launch_slice_t<D, 5>(ctx, sa, raw, grid, s);
    case 6: return launch_slice_t<D, 6>(ctx, sa, raw, grid, s);
    case 7: return launch_slice_t<D, 7>(ctx, sa, raw, grid, s);
    case 8: return launch_slice_t<D, 8>(ctx, sa, raw, grid, s);
    case 10: return launch_slice_t<D, 10>(ctx, sa, raw, grid, s);
    case 12: return launch_slice_t<D, 12>(ctx, sa, raw, grid, s);
  }
  return set_error(DEOCT_ERR_INVALID, "bit-sliced evaluator: %d digits", nd);
}
int launch_slice_1(deoct_ctx* ctx, int nd, const SliceArgs& sa, bool raw, int grid, cudaStream_t s);
int launch_slice_2(deoct_ctx* ctx, int nd, const SliceArgs& sa, bool raw, int grid, cudaStream_t s);
int launch_slice_3(deoct_ctx* ctx, int nd, const SliceArgs& sa, bool raw, int grid, cudaStream_t s);
int launch_slice_4(deoct_ctx* ctx, int nd, const SliceArgs& sa, bool raw, int grid, cudaStream_t s);
int launch_slice_5(deoct_ctx* ctx, int nd, const SliceArgs& sa, bool raw, int grid, cudaStream_t s);

}  // namespace slc
}  // namespace deoct
