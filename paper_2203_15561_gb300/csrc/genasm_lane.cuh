// One window of a pair by one lane: edit-distance columns in difference form
// and the traceback over them. Shared by the batched kernel, the server's
// step and the locate step, for windows of up to 32 * VW bases (VW = 1..4
// 32-bit words per vector).
//
// GenASM's row d says which cells have D(i, j) <= d, where D(i, j) is the
// fewest edits that align the pattern suffix P[wp-1-j ..] with a prefix of the
// text T[i ..] (text end free). A lane holds D itself instead, as the vertical
// differences of one column at a time (bit j of VP / VN: D(i, j) - D(i, j-1)
// is +1 / -1) and steps from column i + 1 to column i with the recurrence of
// Myers (J. ACM 46, 1999) in Hyyro's form (2003):
//   D0 = (((Eq & VP) + VP) ^ VP) | Eq | VN     diagonal difference 0
//   HP = VN | ~(D0 | VP),  HN = VP & D0        horizontal difference +1 / -1
//   VP' = (HN << 1) | ~(D0 | (HP << 1)),  VN' = (HP << 1) & D0
// from the column past the text, D(wt, j) = j + 1. A zero shifts in at j = 0:
// the empty pattern costs nothing at any column. d_min = D(0, wp-1).
//
// The traceback needs no rows either: it only visits cells with D(i, j) = d
// (it starts at d_min, and every edge keeps that equality), so at a cell
//   M is possible iff the bases match (then D(i+1, j-1) = d),
//   S iff D(i+1, j-1) = d - 1: bit j of D0 is clear,
//   I iff D(i, j-1) = d - 1: bit j of VP' is set,
//   D iff D(i+1, j) = d - 1: bit j of HP is set,
// the edges that rows d and d-1 show. With M > S > I > D the last test is
// implied, so a column's table entry is D0 and VP'.
//
// Why this form. A column costs 10 word operations per 32 rows whatever d_min
// is; the row form costs 6 per cell and row (2,112 cells of a random 64-base
// window: 12,700 against 1,300 for its 64 columns). One lane runs a window
// alone, so a warp runs 32 windows with no shuffle, vote or ramp in the
// recurrence, and the walk is one lane's as well: 32 walks per warp instead
// of 4. A table entry is 16 bytes of a 64-row column instead of 4-8 bytes per
// row. Bound: the integer ALU pipe (see the kernels for what it measured).
//
// Every lane keeps to its own shared-memory words (word index * 32 + lane),
// so all accesses are free of bank conflicts and no lane waits for another;
// the warp reconverges at window boundaries only so that its lanes issue
// together.
#pragma once

#include <cstdint>

#include "genasm_internal.h"
#include "genasm_window.cuh"
#include "genasm_words.h"

namespace ga {

// Places that a walk in an order with I or D before M looks at along the diagonal
// for edges that come before M. (An op an iteration took one pair of 10 kb without
// errors 1,280 us; 4 places 885, 8 846, but 8 take one of sequences that do not match
// 1,567 instead of 1,420.)
constexpr int kWalkAhead = 4;

// A warp of LP pairs with NL lanes each. One lane per pair: LP = 32, or 16
// (half a warp) where the tables of 32 would leave schedulers without a warp.
// Several: LP * NL = 32, lane q of a pair holds word q of the vectors.
//
// Shared memory of a warp. Eq: four masks per lane, of all words or its own.
// Table: per stored column {D0, VP'}, then (orders other than the default) HP;
// the words of a column together where one lane has two of them, else apart.
// Planes (VW >= 3): the low and high code bits of the window's read and
// reference bases, VW words and a zero each.
template <int VW, int LP, int NL>
struct LaneShape {
  static constexpr int kThreads = LP * NL;
  static constexpr uint32_t kMask = kThreads == 32 ? 0xffffffffu : (1u << (kThreads & 31)) - 1u;
  static_assert(NL == 1 || NL == 4, "one lane per pair or four");
  // The first lane of each pair.
  static constexpr uint32_t kLeaders = kMask & (NL == 1 ? 0xffffffffu : 0x11111111u);
  static constexpr int kEqWords = NL > 1 ? 1 : VW;  // per lane and mask
  static constexpr uint32_t kEqLane = kEqWords == 1 ? 4u : kEqWords == 2 ? 8u : 16u;
  static constexpr uint32_t kEqRow = 32u * kEqLane;  // a power of two: 128, 256 or 512
  static constexpr uint32_t kEqBytes = 4u * kEqRow;
  static constexpr uint32_t kWord = 4u * LP;            // one word of every pair
  static constexpr uint32_t kPlane = (VW + 1) * kWord;  // one plane
  static constexpr uint32_t kPlaneBytes = VW >= 3 ? 4u * kPlane : 0u;
  static constexpr uint32_t kColBytes = VW * 2u * kWord;  // {D0, VP'} of one column
  static constexpr uint32_t kHpBytes = VW * kWord;        // HP of one column
  static constexpr bool kTogether = VW == 2 && NL == 1;
  // Staged kernels (VW <= 2): the packed words that the next window's bases can
  // lie in, of the read and the reference, copied one window ahead.
  static constexpr uint32_t kStageSeq = (4 * VW + 1) * 128u;
  static constexpr uint32_t kPairBytes = kTogether ? 16u : 8u;  // a pair's entry (or its word's)
  // Columns past the stored ones: one that a walk may look at, and those that
  // the lanes of a pair run ahead of its first lane.
  static constexpr int kSpare = 1 + 2 * (NL - 1);
  // The warp's bytes with tables of `cols` columns.
  static constexpr size_t bytes(int cols, bool any_order, bool staged) {
    return kEqBytes + kPlaneBytes + (staged ? 2u * kStageSeq : 0u) +
           static_cast<size_t>(cols + kSpare) * (kColBytes + (any_order ? kHpBytes : 0u));
  }
};

// A pair in the hands of a lane.
template <int VW>
struct LanePair {
  const uint8_t* read;
  const uint8_t* ref;
  uint32_t* out;      // its CIGAR runs
  uint64_t cells;
  uint32_t cap;       // room for runs (0 in the lanes that do not write them, see `room`)
  uint32_t room;      // the pair's room for runs
  // The open run, and its place in `out`. A pair starts with a run of no
  // length at place -1, which no capacity lets be stored.
  uint32_t run_at, run_op, run_len;
  uint32_t pair, m, n, pos_p, pos_t, edits, windows;
  int32_t status;
  bool busy;
  // The next window's bases: staged from the word at the low address bits
  // p_word / t_word on, or loading.
  uint32_t p_word, t_word;
  uint32_t pw[2 * VW + 1], tw[2 * VW + 1];
};

__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t x) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ void sts64(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

// Asynchronous copy of a word from global to shared memory, and the wait for all
// of this lane's.
__device__ __forceinline__ void copy_word(uint32_t to, const uint32_t* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(from) : "memory");
}
__device__ __forceinline__ void copies_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One Eq mask of VW words (read-only between window starts).
template <int VW>
__device__ __forceinline__ void load_eq(uint32_t a, uint32_t (&e)[VW]) {
  if constexpr (VW == 1) {
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(e[0]) : "r"(a));
  } else if constexpr (VW == 2) {
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(e[0]), "=r"(e[1]) : "r"(a));
  } else if constexpr (VW == 3) {
    uint32_t z;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(e[0]), "=r"(e[1]), "=r"(e[2]), "=r"(z) : "r"(a));
  } else {
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(e[0]), "=r"(e[1]), "=r"(e[2]), "=r"(e[3]) : "r"(a));
  }
}

__device__ __forceinline__ void sts128(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
  asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w)
               : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}

// s = a + b over VW words (the carry out of the top word is dropped).
template <int VW>
__device__ __forceinline__ void add_words(const uint32_t (&a)[VW], const uint32_t (&b)[VW],
                                          uint32_t (&s)[VW]) {
  if constexpr (VW == 1) {
    s[0] = a[0] + b[0];
  } else if constexpr (VW == 2) {
    asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;"
        : "=r"(s[0]), "=r"(s[1]) : "r"(a[0]), "r"(a[1]), "r"(b[0]), "r"(b[1]));
  } else if constexpr (VW == 3) {
    asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(b[0]), "r"(b[1]), "r"(b[2]));
  } else {
    asm("add.cc.u32 %0, %4, %8;\n\taddc.cc.u32 %1, %5, %9;\n\taddc.cc.u32 %2, %6, %10;\n\t"
        "addc.u32 %3, %7, %11;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]));
  }
}

// One column: VP, VN of column i + 1 become those of column i; D0 and HP are
// column i's.
template <int VW>
__device__ __forceinline__ void column_step(const uint32_t (&eq)[VW], uint32_t (&vp)[VW],
                                            uint32_t (&vn)[VW], uint32_t (&d0)[VW],
                                            uint32_t (&hp)[VW], uint32_t (&hn)[VW]) {
  uint32_t t[VW], s[VW];
#pragma unroll
  for (int k = 0; k < VW; ++k) t[k] = eq[k] & vp[k];
  add_words<VW>(t, vp, s);
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    const uint32_t x = eq[k] | vn[k];
    d0[k] = (s[k] ^ vp[k]) | x;
    hp[k] = vn[k] | ~(d0[k] | vp[k]);
    hn[k] = vp[k] & d0[k];
  }
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    const uint32_t hps = k ? __funnelshift_l(hp[k - 1], hp[k], 1) : hp[0] << 1;
    const uint32_t hns = k ? __funnelshift_l(hn[k - 1], hn[k], 1) : hn[0] << 1;
    vp[k] = hns | ~(d0[k] | hps);
    vn[k] = hps & d0[k];
  }
}

// The aligned words that hold the 32 * VW bases at `pos` of a packed sequence of
// `len` bases. Only words that hold a base of the sequence are read.
template <int VW>
__device__ __forceinline__ void load_words(const uint8_t* seq, uint32_t len, uint32_t pos,
                                           uint32_t (&x)[2 * VW + 1]) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(seq) + (pos >> 2);
  const uint32_t* wa = reinterpret_cast<const uint32_t*>(a & ~static_cast<uintptr_t>(3));
  const uint32_t o = 8u * static_cast<uint32_t>(a & 3u) + 2u * (pos & 3u);
  const uint32_t end = bases_end(o, len, pos, 32u * VW);
#pragma unroll
  for (int k = 0; k <= 2 * VW; ++k) x[k] = holds_base(k, o, end) ? __ldg(wa + k) : 0u;
}

// Starts copying the words from base `pos` on that hold its window's bases and
// those of any window up to 32 * VW bases further to shared memory (one word of
// every lane to 128 bytes). Only words that hold a base of the sequence are read.
template <int VW>
__device__ __forceinline__ uint32_t stage_words(const uint8_t* seq, uint32_t len, uint32_t pos, uint32_t to) {
  constexpr int kWords = 4 * VW + 1;
  const uintptr_t a = reinterpret_cast<uintptr_t>(seq) + (pos >> 2);
  const uint32_t* wa = reinterpret_cast<const uint32_t*>(a & ~static_cast<uintptr_t>(3));
  const uint32_t o = 8u * static_cast<uint32_t>(a & 3u) + 2u * (pos & 3u);
  const uint32_t end = bases_end(o, len, pos, 16u * kWords);
  if (end >= 32u * kWords) {
#pragma unroll
    for (int k = 0; k < kWords; ++k) copy_word(to + 128u * k, wa + k);
  } else {
#pragma unroll
    for (int k = 0; k < kWords; ++k)
      if (holds_base(k, o, end)) copy_word(to + 128u * k, wa + k);
  }
  return static_cast<uint32_t>(a) & ~3u;
}

__device__ __forceinline__ uint32_t lo_word(const uint8_t* seq) {
  return static_cast<uint32_t>(reinterpret_cast<uintptr_t>(seq)) & ~3u;
}

// The staged words of the window at `pos` (`word`: what stage_words returned).
template <int VW>
__device__ __forceinline__ void staged_words(const uint8_t* seq, uint32_t pos, uint32_t word, uint32_t from,
                                             uint32_t (&x)[2 * VW + 1]) {
  const uint32_t a = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(seq) + (pos >> 2)) & ~3u;
  const uint32_t at = from + (a - word) * 32u;  // four bytes further on: 128 bytes
#pragma unroll
  for (int k = 0; k <= 2 * VW; ++k) x[k] = lds32(at + 128u * k);
}

// The bases themselves, 16 per word (past the end of the sequence: anything).
template <int VW>
__device__ __forceinline__ void align_bases(const uint8_t* seq, uint32_t pos,
                                            const uint32_t (&x)[2 * VW + 1], uint32_t (&w)[2 * VW]) {
  const uint32_t o = 8u * (static_cast<uint32_t>(reinterpret_cast<uintptr_t>(seq) + (pos >> 2)) & 3u) +
                     2u * (pos & 3u);
#pragma unroll
  for (int k = 0; k < 2 * VW; ++k) w[k] = __funnelshift_r(x[k], x[k + 1], o);
}

// Low and high code bits of the bases in `w`: bit 31 - u of word k of L / H is
// base 32k + u's.
template <int VW>
__device__ __forceinline__ void bit_planes(const uint32_t (&w)[2 * VW], uint32_t (&L)[VW],
                                           uint32_t (&H)[VW]) {
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    uint32_t u[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      // Delta swaps gather each byte pair's even bits in its low byte and its
      // odd bits in its high byte.
      uint32_t x = w[2 * k + q], t;
      t = (x ^ (x >> 1)) & 0x22222222u;
      x ^= t ^ (t << 1);
      t = (x ^ (x >> 2)) & 0x0C0C0C0Cu;
      x ^= t ^ (t << 2);
      t = (x ^ (x >> 4)) & 0x00F000F0u;
      x ^= t ^ (t << 4);
      u[q] = x;
    }
    L[k] = __brev(__byte_perm(u[0], u[1], 0x6420));
    H[k] = __brev(__byte_perm(u[0], u[1], 0x7531));
  }
}

// Eq masks (bit j set iff P[wp-1-j] is the base) from the pattern's planes,
// into the lane's Eq words: all of them, or (several lanes per pair) word q.
// Bits at and above wp: anything.
template <int VW, int LP, int NL>
__device__ __forceinline__ void store_eq(uint32_t eq_lane, uint32_t q, int wp, const uint32_t (&L)[VW],
                                         const uint32_t (&H)[VW]) {
  // As one number, bit j is base 32*VW-1-j's: down by 32*VW - wp bits.
  uint32_t l[VW], h[VW];
  const uint32_t sh = static_cast<uint32_t>(32 * VW - wp);
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    l[k] = L[VW - 1 - k];
    h[k] = H[VW - 1 - k];
  }
#pragma unroll
  for (int b = VW > 2 ? 64 : 32; b >= 32; b >>= 1) {  // whole words
    const bool by = (sh & static_cast<uint32_t>(b)) != 0;
#pragma unroll
    for (int k = 0; k < VW; ++k) {
      const int from = k + b / 32;
      l[k] = by ? (from < VW ? l[from] : 0u) : l[k];
      h[k] = by ? (from < VW ? h[from] : 0u) : h[k];
    }
  }
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    l[k] = __funnelshift_r(l[k], k + 1 < VW ? l[k + 1] : 0u, sh);
    h[k] = __funnelshift_r(h[k], k + 1 < VW ? h[k + 1] : 0u, sh);
  }
  if constexpr (NL > 1) {
#pragma unroll
    for (int k = 1; k < VW; ++k) {
      l[0] = q == static_cast<uint32_t>(k) ? l[k] : l[0];
      h[0] = q == static_cast<uint32_t>(k) ? h[k] : h[0];
    }
  }
  using Shape = LaneShape<VW, LP, NL>;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint32_t e[VW];
#pragma unroll
    for (int k = 0; k < Shape::kEqWords; ++k)
      e[k] = (c & 1 ? l[k] : ~l[k]) & (c & 2 ? h[k] : ~h[k]);
    const uint32_t a = eq_lane + c * Shape::kEqRow;
    if constexpr (Shape::kEqWords == 1) {
      sts32(a, e[0]);
    } else {
      sts64(a, e[0], e[1]);
      if constexpr (Shape::kEqWords == 3) sts32(a + 8, e[2]);
      if constexpr (Shape::kEqWords == 4) sts64(a + 8, e[VW - 2], e[VW - 1]);
    }
  }
}

// Address of the Eq masks (EW words each) of base x of a word of text bases.
template <int EW>
__device__ __forceinline__ uint32_t eq_at(uint32_t eq_lane, uint32_t tw, int x) {
  constexpr int kLog = EW == 1 ? 7 : EW == 2 ? 8 : 9;  // bytes of the row of a base
  const int sh = 2 * x - kLog;
  const uint32_t c = sh >= 0 ? tw >> sh : tw << -sh;
  return eq_lane | (c & (3u << kLog));
}

// The Eq masks of bases x0 + 7 .. x0 of a word of text bases.
template <int EW>
__device__ __forceinline__ void load_eq8(uint32_t eq_lane, uint32_t tw, int x0,
                                         uint32_t (&e)[8][EW]) {
#pragma unroll
  for (int x = 7; x >= 0; --x) load_eq<EW>(eq_at<EW>(eq_lane, tw, x0 + x), e[x]);
}

// Eight columns, right to left from column c0 + 7, c0 of the window; their
// table entries go to `row` (column c0's) when `keep` is set.
template <int VW, int LP, bool kMask, bool kHp>
__device__ __forceinline__ void eight_columns(const uint32_t (&e)[8][VW], int left, bool keep,
                                              uint32_t row, uint32_t hrow, uint32_t (&vp)[VW],
                                              uint32_t (&vn)[VW]) {
  using Shape = LaneShape<VW, LP, 1>;
#pragma unroll
  for (int x = 7; x >= 0; --x) {
    uint32_t eq[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) eq[k] = kMask && x >= left ? 0u : e[x][k];
    uint32_t d0[VW], hp[VW], hn[VW];
    column_step<VW>(eq, vp, vn, d0, hp, hn);
    if (keep) {
      const uint32_t at = row + x * Shape::kColBytes;
      if constexpr (Shape::kTogether) {
        sts128(at, d0[0], d0[VW - 1], vp[0], vp[VW - 1]);
      } else {
#pragma unroll
        for (int k = 0; k < VW; ++k) sts64(at + k * 2 * Shape::kWord, d0[k], vp[k]);
      }
#pragma unroll
      for (int k = 0; k < VW; ++k)
        if constexpr (kHp) sts32(hrow + x * Shape::kHpBytes + k * Shape::kWord, hp[k]);
    }
  }
}

// D(0, wp-1) from the differences of column 0 (word k of the vectors).
__device__ __forceinline__ int word_distance(int wp, int k, uint32_t vp, uint32_t vn) {
  const int bits = wp - 32 * k;
  const uint32_t mask = bits >= 32 ? ~0u : bits > 0 ? (1u << bits) - 1u : 0u;
  return __popc(vp & mask) - __popc(vn & mask);
}

// The columns of a window by one lane, right to left from column 16 * ncols16 -
// 1: the table entries of columns [cb, end) (cb a multiple of 8, `end` rounded up
// to one) go to `tab_lane`. With kMask, columns at and past wt leave the initial
// column as it is (no base matches there: D(wt, j) = j + 1 repeats). Returns
// D(0, wp-1). The Eq masks are loaded eight columns ahead, before the stores of
// the columns in between: the recurrence itself never waits for shared memory.
template <int VW, int LP, bool kMask, bool kHp>
__device__ __forceinline__ int window_columns(int wp, int wt, int ncols16, uint32_t (&tw)[2 * VW],
                                              uint32_t eq_lane, uint32_t tab_lane, uint32_t hp_lane,
                                              int cb, int end) {
  using Shape = LaneShape<VW, LP, 1>;
  uint32_t vp[VW], vn[VW];
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    vp[k] = ~0u;
    vn[k] = 0u;
  }
  // The text words move up so that the next one to use is always the last.
  for (int b = 2 * VW; b > ncols16; --b) {
#pragma unroll
    for (int k = 2 * VW - 1; k > 0; --k) tw[k] = tw[k - 1];
  }
  uint32_t hi[8][VW], lo[8][VW];
  load_eq8<VW>(eq_lane, tw[2 * VW - 1], 8, hi);
  uint32_t row = tab_lane + static_cast<uint32_t>(16 * ncols16 - cb) * Shape::kColBytes;
  uint32_t hrow = hp_lane + static_cast<uint32_t>(16 * ncols16 - cb) * Shape::kHpBytes;
  for (int c0 = 16 * ncols16 - 16; c0 >= 0; c0 -= 16) {
    load_eq8<VW>(eq_lane, tw[2 * VW - 1], 0, lo);
    row -= 16u * Shape::kColBytes;
    hrow -= 16u * Shape::kHpBytes;
    eight_columns<VW, LP, kMask, kHp>(hi, wt - c0 - 8, c0 + 8 >= cb && c0 + 8 < end,
                                      row + 8u * Shape::kColBytes, hrow + 8u * Shape::kHpBytes, vp, vn);
#pragma unroll
    for (int k = 2 * VW - 1; k > 0; --k) tw[k] = tw[k - 1];
    load_eq8<VW>(eq_lane, tw[2 * VW - 1], 8, hi);  // (past the last block: not used)
    eight_columns<VW, LP, kMask, kHp>(lo, wt - c0, c0 >= cb && c0 < end, row, hrow, vp, vn);
  }
  int d = 0;
#pragma unroll
  for (int k = 0; k < VW; ++k) d += word_distance(wp, k, vp[k], vn[k]);
  return d;
}

// The columns of a window by the NL lanes of a pair, lane q word q of each
// vector. Lane q is two columns behind lane q - 1, which sends it what its word
// hands up (the carry of the addition and the two bits shifted out) by shuffle:
// sent at the end of a step and used two steps later, they have arrived by
// then. A step is one word's eleven operations and the three shuffles whatever
// the width: 49 cycles for one warp per scheduler, against 47 for a column of
// two words by one lane and 95 of four.
struct WordLink {
  uint32_t carry, hp, hn;
};

template <int VW, int LP, int NL, bool kHp>
struct SplitColumns {
  using Shape = LaneShape<VW, LP, NL>;
  uint32_t vp, vn;
  WordLink next, after;  // from lane q - 1: for this step and the one after it
  uint32_t top_bit;      // 31, and 32 for lane 0 (which gets nothing from below)
  bool stores;           // a lane that has a word

  __device__ __forceinline__ void step(uint32_t eq, bool on, bool keep, uint32_t at, uint32_t hat) {
    const uint32_t in = __funnelshift_rc(next.carry, 0u, top_bit);
    const uint32_t hin = __funnelshift_rc(next.hp, 0u, top_bit);
    const uint32_t gin = __funnelshift_rc(next.hn, 0u, top_bit);
    const uint32_t t = eq & vp;
    const uint32_t s = t + vp + in;
    const uint32_t a = (s ^ vp) | eq;
    const uint32_t h = vn | ~(a | vp);
    const uint32_t g = vp & a;
    const uint32_t d0 = a | vn;
    next = after;
    after.carry = __shfl_up_sync(Shape::kMask, t | (vp & ~s), 1);  // bit 31: the carry out
    after.hp = __shfl_up_sync(Shape::kMask, h, 1);
    after.hn = __shfl_up_sync(Shape::kMask, g, 1);
    const uint32_t hs = h + h + hin, gs = g + g + gin;
    const uint32_t vp1 = gs | ~(d0 | hs), vn1 = hs & d0;
    vp = on ? vp1 : vp;
    vn = on ? vn1 : vn;
    if (keep && on && (NL == VW || stores)) {
      sts64(at, d0, vp);
      if constexpr (kHp) sts32(hat, h);
    }
  }
};

template <int VW, int LP, int NL, bool kMask, bool kHp>
__device__ __forceinline__ int split_columns(uint32_t q, int wp, int wt, int ncols16,
                                             const uint32_t (&tw)[2 * VW], uint32_t eq_lane,
                                             uint32_t tab_lane, uint32_t hp_lane, int end) {
  using Shape = LaneShape<VW, LP, NL>;
  // At word 0's column c this lane is at column c + 2q: its text starts 2q bases
  // in, and column c's row is 2q columns on.
  uint32_t w[2 * VW];
#pragma unroll
  for (int k = 0; k < 2 * VW; ++k)
    w[k] = __funnelshift_r(tw[k], k + 1 < 2 * VW ? tw[k + 1] : 0u, 4u * q);
  const uint32_t tail = q ? tw[0] << (32u - 4u * q) : 0u;  // its first 2q bases, at the top
  const int wt_lane = wt - static_cast<int>(2u * q);
  tab_lane += 2u * q * Shape::kColBytes + q * 2u * Shape::kWord;
  hp_lane += 2u * q * Shape::kHpBytes + q * Shape::kWord;
  SplitColumns<VW, LP, NL, kHp> r;
  r.vp = ~0u;
  r.vn = 0u;
  r.next = r.after = WordLink{0u, 0u, 0u};
  r.top_bit = q ? 31u : 32u;
  r.stores = q < static_cast<uint32_t>(VW);
  for (int b = 2 * VW; b > ncols16; --b) {
#pragma unroll
    for (int k = 2 * VW - 1; k > 0; --k) w[k] = w[k - 1];
  }
  uint32_t hi[8][1], lo[8][1];
  load_eq8<1>(eq_lane, w[2 * VW - 1], 8, hi);
  uint32_t row = tab_lane + static_cast<uint32_t>(16 * ncols16) * Shape::kColBytes;
  uint32_t hrow = hp_lane + static_cast<uint32_t>(16 * ncols16) * Shape::kHpBytes;
  // A lane's first steps, before its own first column, match nothing (its word
  // then stays as it is): the first eight columns are always masked.
  const int cols = 16 * ncols16 - static_cast<int>(2u * q);
  const int left = min(wt_lane, cols);
  const auto mask8 = [&](uint32_t (&e)[8][1], int c) {
#pragma unroll
    for (int x = 0; x < 8; ++x) e[x][0] = c + x < left ? e[x][0] : 0u;
  };
  mask8(hi, 16 * ncols16 - 8);
  for (int c0 = 16 * ncols16 - 16; c0 >= 0; c0 -= 16) {
    load_eq8<1>(eq_lane, w[2 * VW - 1], 0, lo);
    row -= 16u * Shape::kColBytes;
    hrow -= 16u * Shape::kHpBytes;
    const bool keep_hi = c0 + 8 < end, keep_lo = c0 < end;
#pragma unroll
    for (int x = 7; x >= 0; --x)
      r.step(hi[x][0], true, keep_hi, row + (8 + x) * Shape::kColBytes, hrow + (8 + x) * Shape::kHpBytes);
#pragma unroll
    for (int k = 2 * VW - 1; k > 0; --k) w[k] = w[k - 1];
    load_eq8<1>(eq_lane, w[2 * VW - 1], 8, hi);  // (past the last block: not used)
    if constexpr (kMask) {
      mask8(hi, c0 - 8);
      mask8(lo, c0);
    }
#pragma unroll
    for (int x = 7; x >= 0; --x)
      r.step(lo[x][0], true, keep_lo, row + x * Shape::kColBytes, hrow + x * Shape::kHpBytes);
  }
  // The last columns of the lanes behind lane 0.
#pragma unroll
  for (int k = 0; k < 2 * (NL - 1); ++k) {
    const bool on = k < static_cast<int>(2u * q);
    uint32_t e[1];
    load_eq<1>(eq_at<1>(eq_lane, tail, 15 - k), e);
    const bool in = static_cast<int>(2u * q) - 1 - k < wt;
    r.step(in ? e[0] : 0u, on, true, row - (k + 1) * Shape::kColBytes, hrow - (k + 1) * Shape::kHpBytes);
  }
  int d = word_distance(wp, static_cast<int>(q), r.vp, r.vn);
#pragma unroll
  for (int k = 1; k < NL; k <<= 1) d += __shfl_xor_sync(Shape::kMask, d, k);
  return d;
}

// Closes the open run when `when` is set (a run past the capacity is not stored).
template <int VW>
__device__ __forceinline__ void close_run(LanePair<VW>& st, bool when) {
  stg32_if(when && st.run_at < st.cap, st.out + st.run_at, st.run_len << 4 | st.run_op);
  st.run_at += when ? 1u : 0u;
  st.run_len = when ? 0u : st.run_len;
}

// Position of the highest set bit counted from bit 31 (0xffffffff for x = 0).
__device__ __forceinline__ uint32_t leading_zeros(uint32_t x) {
  uint32_t r;
  asm("bfind.shiftamt.u32 %0, %1;" : "=r"(r) : "r"(x));
  return r;
}

// The 32 base bits from position c on (base c in bit 31) of a plane whose word
// k holds bases 32k (bit 31) .. 32k + 31 (bit 0); c <= 32 * VW.
template <int VW, int LP, int NL>
__device__ __forceinline__ uint32_t plane_at(const uint32_t (&w)[VW], uint32_t plane_lane, int which,
                                             uint32_t c) {
  if constexpr (VW == 1) {
    return w[0] << (c & 31u);
  } else if constexpr (VW == 2) {
    const uint64_t x = (static_cast<uint64_t>(w[0]) << 32) | w[1];
    return static_cast<uint32_t>((x << (c & 63u)) >> 32);
  } else {
    using Shape = LaneShape<VW, LP, NL>;
    const uint32_t a = plane_lane + which * Shape::kPlane + min(c >> 5, VW - 1u) * Shape::kWord;
    return __funnelshift_l(lds32(a + Shape::kWord), lds32(a), c);
  }
}

// Bits j of D0 and VP' of a column (at bit 0; other bits: anything). For the
// j = -1 of a finished lane: anything.
template <int VW, int LP, int NL>
__device__ __forceinline__ uint2 column_bits(uint32_t tab0, uint32_t ct, uint32_t j) {
  using Shape = LaneShape<VW, LP, NL>;
  const uint32_t at = tab0 + ct * Shape::kColBytes;
  if constexpr (VW == 1) {
    const uint2 e = lds64(at);
    return make_uint2(e.x >> (j & 31u), e.y >> (j & 31u));
  } else if constexpr (Shape::kTogether) {
    const uint4 e = lds128(at);
    const uint64_t d = (static_cast<uint64_t>(e.y) << 32) | e.x, v = (static_cast<uint64_t>(e.w) << 32) | e.z;
    return make_uint2(static_cast<uint32_t>(d >> (j & 63u)), static_cast<uint32_t>(v >> (j & 63u)));
  } else {
    const uint32_t k = VW == 3 ? min(j >> 5, 2u) : (j >> 5) & (VW - 1u);
    const uint2 e = lds64(at + k * (2u * Shape::kWord));
    return make_uint2(e.x >> (j & 31u), e.y >> (j & 31u));
  }
}

// Bit j of a column's HP, likewise.
template <int VW, int LP, int NL>
__device__ __forceinline__ uint32_t hp_bit(uint32_t hp0, uint32_t ct, uint32_t j) {
  using Shape = LaneShape<VW, LP, NL>;
  const uint32_t k = VW == 3 ? min(j >> 5, 2u) : (j >> 5) & (VW - 1u);
  return lds32(hp0 + ct * Shape::kHpBytes + k * Shape::kWord) >> (j & 31u);
}

// What a walk reads: the window's bit planes and the table's columns.
template <int VW, int LP, int NL>
struct Walk {
  uint32_t pl[VW], ph[VW], tl[VW], th[VW];
  uint32_t plane_lane;
  uint32_t tab0, hp0;  // column 0's entries
  uint32_t top;        // wp - 1
  // Orders other than the default: all ones if I, D come before M; the spare column's HP.
  uint32_t over_i, over_d, hp_end;
  // Where the bases from read position cp and reference position ct on differ
  // (bit 31: the first of them).
  __device__ __forceinline__ uint32_t differ(uint32_t cp, uint32_t ct) const {
    return (plane_at<VW, LP, NL>(pl, plane_lane, 0, cp) ^ plane_at<VW, LP, NL>(tl, plane_lane, 2, ct)) |
           (plane_at<VW, LP, NL>(ph, plane_lane, 1, cp) ^ plane_at<VW, LP, NL>(th, plane_lane, 3, ct));
  }
  // Where along the diagonal from there an insertion or a deletion that comes before
  // M is possible (bit 31: the first place), kWalkAhead places. Bit j - u of column
  // ct + u is turned to bit 31 - u by the same distance whatever u is. (Places past
  // the window's end give anything: past the spare column HP's words are read for
  // columns, of which the table has eight at least, and its last one for HP.)
  __device__ __forceinline__ uint32_t before_match(uint32_t cp, uint32_t ct) const {
    using Shape = LaneShape<VW, LP, NL>;
    const uint32_t j = top - cp;
    const uint32_t vp = tab0 + ct * Shape::kColBytes + (Shape::kTogether ? 8u : 4u), hp = hp0 + ct * Shape::kHpBytes;
    uint32_t found = 0;
#pragma unroll
    for (int u = 0; u < kWalkAhead; ++u) {
      uint32_t k = 0;  // its word
      if constexpr (VW == 2) k = j >= 32u + static_cast<uint32_t>(u) ? 1u : 0u;
      if constexpr (VW == 3) k = min((j - u) >> 5, 2u);
      if constexpr (VW == 4) k = ((j - u) >> 5) & 3u;
      const uint32_t v = lds32(vp + u * Shape::kColBytes + k * (Shape::kTogether ? 4u : 2u * Shape::kWord));
      const uint32_t h = lds32(min(hp + u * Shape::kHpBytes, hp_end) + k * Shape::kWord);
      const uint32_t x = (v & over_i) | (h & over_d);
      found |= __funnelshift_r(x, x, j + 1u) & (0x80000000u >> u);
    }
    return found;
  }
};

// The ops of an iteration: matches, then an edit (0: none). They join the runs
// in the next iteration, once it has asked for its column: the bookkeeping then
// fills the wait for that read instead of standing before it (10,000 pairs of
// 10 kb: 1.133 ms, with it 1.119; one pair 644 us, with it 638).
struct LateOps {
  uint32_t matches, edit;
};
template <class Runs>
__device__ __forceinline__ void book_ops(Runs& st, const LateOps& o) {
  close_run(st, o.matches > 0u && st.run_op != kOpMatch);
  st.run_op = o.matches > 0u ? kOpMatch : st.run_op;
  st.run_len += o.matches;
  close_run(st, o.edit != 0u && st.run_op != o.edit);
  st.run_op = o.edit ? o.edit : st.run_op;
  st.run_len += o.edit ? 1u : 0u;
}

// One iteration of a walk at read base cp and text base ct of the window, up to
// `goal` and `tend`: the matches ahead (up to 32 base pairs compared at once) and
// the edit that ends them. No branches: a lane whose counts are used up appends
// nothing.
template <int VW, int LP, int NL, class Runs>
__device__ __forceinline__ void walk_step(const Walk<VW, LP, NL>& w, Runs& st, uint32_t& cp, uint32_t& ct,
                                          uint32_t goal, uint32_t tend, LateOps& late) {
  const uint32_t lim = min(min(goal - cp, tend - ct), 32u);
  const uint32_t z = leading_zeros(w.differ(cp, ct));
  const uint32_t L = min(z, lim);
  const uint32_t one = z < lim ? 1u : 0u;  // an edit ends the matches
  cp += L;
  ct += L;
  const uint2 e = column_bits<VW, LP, NL>(w.tab0, ct, w.top - cp);
  book_ops(st, late);
  late.matches = L;
  // S (D0 clear) takes a base of both, I (VP' set) of the read, D of the text.
  const uint32_t from_p = one & (e.y | ~e.x), from_t = one & ~(e.x & e.y);
  const uint32_t code = from_p + 2u * from_t;
  late.edit = code == 3u ? kOpSubst : code;
  st.edits += one;
  cp += from_p;
  ct += from_t;
}

// The same in any other order, as many matches as are sure to be taken and the op
// after them: up to a mismatch, or to where an insertion or a deletion that comes
// before M is possible (a substitution never is where the bases match), kWalkAhead
// places ahead at most.
template <int VW, int LP, int NL>
__device__ __forceinline__ uint32_t any_op(const Walk<VW, LP, NL>& w, uint64_t tb_table, uint32_t cp, uint32_t ct,
                                           uint32_t mm) {
  const uint32_t j = w.top - cp;
  const uint2 e = column_bits<VW, LP, NL>(w.tab0, ct, j);
  const uint32_t h = hp_bit<VW, LP, NL>(w.hp0, ct, j);
  const uint32_t can = (~mm >> 31) << kTbM | (~e.x & 1u) << kTbS | (e.y & 1u) << kTbI | (h & 1u) << kTbD;
  const uint32_t code = static_cast<uint32_t>(tb_table >> (4 * can)) & 15u;
  return (kTbOps >> (4u * code)) & 15u;
}
template <int VW, int LP, int NL, class Runs>
__device__ __forceinline__ void walk_step_ahead(const Walk<VW, LP, NL>& w, uint64_t tb_table, Runs& st,
                                                uint32_t& cp, uint32_t& ct, uint32_t goal, uint32_t tend) {
  const uint32_t lim = min(min(goal - cp, tend - ct), 32u);
  const uint32_t mm = w.differ(cp, ct);
  uint32_t ends = mm;
  if (w.over_i | w.over_d) ends |= w.before_match(cp, ct) | (0x80000000u >> kWalkAhead);
  const uint32_t z = leading_zeros(ends);
  const uint32_t L = min(z, lim);
  const uint32_t one = z < lim ? 1u : 0u;
  cp += L;
  ct += L;
  const uint32_t op = any_op<VW, LP, NL>(w, tb_table, cp, ct, mm << (L & 31u));
  book_ops(st, LateOps{L, one ? op : 0u});
  st.edits += op != kOpMatch ? one : 0u;
  cp += op != kOpDel ? one : 0u;
  ct += op != kOpIns ? one : 0u;
}

// One op in any order.
template <int VW, int LP, int NL, class Runs>
__device__ __forceinline__ void walk_step_any(const Walk<VW, LP, NL>& w, uint64_t tb_table, Runs& st,
                                              uint32_t& cp, uint32_t& ct, uint32_t goal, uint32_t tend) {
  const uint32_t lim = min(min(goal - cp, tend - ct), 32u);
  const uint32_t one = lim > 0u ? 1u : 0u;
  const uint32_t op = any_op<VW, LP, NL>(w, tb_table, cp, ct, w.differ(cp, ct));
  close_run(st, one != 0u && st.run_op != op);
  st.run_op = one ? op : st.run_op;
  st.run_len += one;
  st.edits += op != kOpMatch ? one : 0u;
  cp += op != kOpDel ? one : 0u;
  ct += op != kOpIns ? one : 0u;
}

// Starts loading the bases of the pair's next window: to shared memory, or into
// registers.
template <int VW, bool kStaged>
__device__ __forceinline__ void lane_fetch(LanePair<VW>& st, uint32_t base) {
  using Shape = LaneShape<VW, 32, 1>;
  if constexpr (kStaged) {
    const uint32_t to = base + Shape::kEqBytes + (threadIdx.x & 31u) * 4u;
    copies_wait();  // of a pair that was put back or failed: no two copies to one place
    st.p_word = stage_words<VW>(st.read, st.m, st.pos_p, to);
    st.t_word = stage_words<VW>(st.ref, st.n, st.pos_t, to + Shape::kStageSeq);
  } else {
    load_words<VW>(st.read, st.m, st.pos_p, st.pw);
    load_words<VW>(st.ref, st.n, st.pos_t, st.tw);
  }
}

// One window of the lane's pair (the window chain of a pair is serial: each
// window starts where the previous traceback stopped; its bases start to load
// there). Lanes without a pair come along with ga false. kAny: traceback orders
// other than M > S > I > D.
//
// The table holds `cols` columns (a multiple of 8); a traceback that walks
// past them has the columns computed again with the next `cols` stored. With
// several lanes per pair it holds them all; the lanes walk together, each with
// the pair's whole state, and the first one writes its runs.
//
// kStaged: the packed words of the next window are copied to shared memory while
// this one is computed; otherwise they are loaded into registers once its walk
// has ended. With many pairs per warp some lane's load goes to L2 or further in
// nearly every window (10,000 pairs of 10 kb: 1.21 ms, staged 1.14); a pair alone
// in its warp, or two warps per scheduler, wait little and save the copies'
// instructions (one pair 633 us, staged 660).
template <int VW, int LP, int NL, bool kAny, bool kStaged>
__device__ __forceinline__ void lane_window(const AlignParams& p, LanePair<VW>& st, uint32_t base,
                                            int cols) {
  using Shape = LaneShape<VW, LP, NL>;
  constexpr uint32_t kMask = Shape::kMask;
  // Another order than the default: whether windows of few edits (every lane's) walk
  // by matches. One pair of 10 kb, DIMS, without errors: 885 us, an op an iteration
  // 1,285; at 10% errors 1,080, 1,312. Windows of many edits gain nothing by it (one
  // pair that does not match: 1,420 us against 1,310), and wide windows by one lane
  // each lose in both forms to the larger kernel (5,000 pairs at W = 128 7%).
  constexpr bool kAhead = VW <= 2 || NL > 1;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t q = lane % NL, slot = lane / NL;
  const uint32_t eq_lane = base + lane * Shape::kEqLane;
  constexpr uint32_t kStageBytes = kStaged ? 2u * Shape::kStageSeq : 0u;
  const uint32_t tab_base = base + Shape::kEqBytes + kStageBytes + Shape::kPlaneBytes;
  const uint32_t tab_lane = tab_base + slot * Shape::kPairBytes;
  const uint32_t hp_lane =
      tab_base + static_cast<uint32_t>(cols + Shape::kSpare) * Shape::kColBytes + slot * 4u;
  const bool ga = st.busy;
  const int commit = p.W - p.O;
  int wp = 1, wt = 0;
  if (ga) {
    wp = static_cast<int>(min(static_cast<uint32_t>(p.W), st.m - st.pos_p));
    wt = static_cast<int>(min(static_cast<uint32_t>(p.W), st.n - st.pos_t));
  }
  const bool last = !ga || st.pos_p + static_cast<uint32_t>(wp) == st.m;
  Walk<VW, LP, NL> w;
  uint32_t tw[2 * VW];
  {
    uint32_t pw[2 * VW];
    if constexpr (kStaged) {
      // (a lane without a pair reads its first words)
      const uint32_t from = base + Shape::kEqBytes + lane * 4u;
      copies_wait();
      staged_words<VW>(st.read, ga ? st.pos_p : 0u, ga ? st.p_word : lo_word(st.read), from, st.pw);
      staged_words<VW>(st.ref, ga ? st.pos_t : 0u, ga ? st.t_word : lo_word(st.ref),
                       from + Shape::kStageSeq, st.tw);
    }
    align_bases<VW>(st.read, st.pos_p, st.pw, pw);
    align_bases<VW>(st.ref, st.pos_t, st.tw, tw);
    bit_planes<VW>(pw, w.pl, w.ph);
    bit_planes<VW>(tw, w.tl, w.th);
  }
  // The next window starts W - O bases further at most: its words, while this
  // window is computed. (This window's have been used: the planes depend on them.)
  if constexpr (kStaged) {
    if (ga && !last) lane_fetch<VW, true>(st, base);
  }
  store_eq<VW, LP, NL>(eq_lane, q, wp, w.pl, w.ph);
  w.plane_lane = base + Shape::kEqBytes + kStageBytes + slot * 4u;
  if constexpr (VW >= 3) {
#pragma unroll
    for (int k = 0; k <= VW; ++k) {
      const uint32_t a = w.plane_lane + k * Shape::kWord;
      sts32(a, k < VW ? w.pl[k < VW ? k : 0] : 0u);
      sts32(a + Shape::kPlane, k < VW ? w.ph[k < VW ? k : 0] : 0u);
      sts32(a + 2u * Shape::kPlane, k < VW ? w.tl[k < VW ? k : 0] : 0u);
      sts32(a + 3u * Shape::kPlane, k < VW ? w.th[k < VW ? k : 0] : 0u);
    }
  }
  w.top = static_cast<uint32_t>(wp) - 1u;
  if constexpr (kAny) {  // what the table takes of {M, I} and of {M, D}
    w.over_i = (p.tb_table >> (4 * (1 << kTbM | 1 << kTbI)) & 15u) == kTbI ? ~0u : 0u;
    w.over_d = (p.tb_table >> (4 * (1 << kTbM | 1 << kTbD)) & 15u) == kTbD ? ~0u : 0u;
    w.hp_end = hp_lane + static_cast<uint32_t>(cols) * Shape::kHpBytes;
  }
  const int ncols16 = (p.W + 15) >> 4;
  // A window that stops W - O bases in, before its text can run out, ends when
  // either count gets there; others end with their pattern bases (the text
  // used up: only insertions are left).
  const bool inner = !last && commit <= wt;
  uint32_t goal = !ga ? 0u : static_cast<uint32_t>(last ? wp : commit);  // pattern bases to take
  const uint32_t text = static_cast<uint32_t>(inner ? commit : wt);      // text bases it may take
  uint32_t cp = 0, ct = 0;
  int dmin = -1;
  // Some lane's text or pattern ends here: masked columns, and walks that can
  // reach all of them.
  const bool mask = __any_sync(kMask, ga && (wt < 16 * ncols16 || !inner));
  const int need = mask ? 32 * VW : commit;
  for (int cb = 0;; cb += cols) {
    uint32_t t2[2 * VW];
#pragma unroll
    for (int k = 0; k < 2 * VW; ++k) t2[k] = tw[k];
    const int end = min(cb + cols, need);
    int d;
    if constexpr (NL == 1) {
      d = mask ? window_columns<VW, LP, true, kAny>(wp, wt, ncols16, t2, eq_lane, tab_lane, hp_lane,
                                                    cb, end)
               : window_columns<VW, LP, false, kAny>(wp, wt, ncols16, t2, eq_lane, tab_lane, hp_lane,
                                                     cb, end);
    } else {
      __syncwarp(kMask);  // the walks of the window before are over
      d = mask ? split_columns<VW, LP, NL, true, kAny>(q, wp, wt, ncols16, t2, eq_lane, tab_lane,
                                                       hp_lane, end)
               : split_columns<VW, LP, NL, false, kAny>(q, wp, wt, ncols16, t2, eq_lane, tab_lane,
                                                        hp_lane, end);
      __syncwarp(kMask);  // the other lanes' words are in the table
    }
    if (cb == 0) {
      dmin = d;
      if (dmin > p.kmax) goal = 0u;
    }
    // A lane that walks in this pass stands at column cb, the others stay put
    // wherever they are (their reads go to column 0 of the table). Text bases of
    // this pass: up to the stored columns' end (the table has a spare one there).
    const bool walks = cp < goal && ct < text;
    const uint32_t at0 = walks ? static_cast<uint32_t>(cb) : ct;
    const uint32_t tend = walks ? min(text, static_cast<uint32_t>(cb + cols)) : ct;
    w.tab0 = tab_lane - at0 * Shape::kColBytes;
    w.hp0 = hp_lane - at0 * Shape::kHpBytes;
    LateOps late{0u, 0u};
    // Each lane on its own until its counts are used up: a vote of the warp per
    // round costs more than the lanes that wait for the longest walk. Two
    // iterations to a test.
    if constexpr (!kAny) {
      while (cp < goal && ct < tend) {
        walk_step<VW, LP, NL>(w, st, cp, ct, goal, tend, late);
        walk_step<VW, LP, NL>(w, st, cp, ct, goal, tend, late);
      }
      book_ops(st, late);
    } else if (kAhead && __all_sync(kMask, (w.over_i | w.over_d) == 0u || !ga || 8 * dmin <= p.W)) {
      while (cp < goal && ct < tend) {
        walk_step_ahead<VW, LP, NL>(w, p.tb_table, st, cp, ct, goal, tend);
        if constexpr (VW <= 2) walk_step_ahead<VW, LP, NL>(w, p.tb_table, st, cp, ct, goal, tend);
      }
    } else {
      while (cp < goal && ct < tend) {
        walk_step_any<VW, LP, NL>(w, p.tb_table, st, cp, ct, goal, tend);
        walk_step_any<VW, LP, NL>(w, p.tb_table, st, cp, ct, goal, tend);
      }
    }
    __syncwarp(kMask);
    if (cb + cols >= need || !__any_sync(kMask, cp < goal && ct < text)) break;
  }
  if (ga) {
    if (cp < goal && !inner) {  // the text is used up
      close_run(st, st.run_op != kOpIns);
      st.run_op = kOpIns;
      st.run_len += goal - cp;
      st.edits += goal - cp;
      cp = goal;
    }
    if (dmin > p.kmax) {
      st.status = kPairExceedsK;
    } else if (static_cast<int32_t>(st.run_at) >= 0 && st.run_at > st.room) {
      st.status = kPairCigarFull;
    } else {
      ++st.windows;
      st.cells += static_cast<uint64_t>(wt) * static_cast<uint64_t>(dmin + 1);
      st.pos_p += cp;
      st.pos_t += ct;
      if constexpr (!kStaged) {
        if (st.pos_p < st.m) lane_fetch<VW, false>(st, base);
      }
    }
  }
}

// The lane's pair is done once a window ended it or its read is used up.
template <int VW>
__device__ __forceinline__ bool lane_done(const LanePair<VW>& st) {
  return st.status != kPairOk || st.pos_p >= st.m;
}

template <int VW>
__device__ __forceinline__ void lane_finish(const AlignParams& p, LanePair<VW>& st, bool writer) {
  if (st.status == kPairOk && st.run_at != 0xffffffffu) {
    if (st.run_at >= st.room) st.status = kPairCigarFull;
    close_run(st, true);
  }
  st.busy = false;
  if (!writer) return;
  const bool ok = st.status == kPairOk;
  p.dist[st.pair] = ok ? static_cast<int32_t>(st.edits) : -1;
  p.status[st.pair] = st.status;
  p.ref_consumed[st.pair] = ok ? static_cast<int32_t>(st.pos_t) : -1;
  if (p.ref_start && !ok) p.ref_start[st.pair] = -1;
  p.n_runs[st.pair] = ok && st.run_at != 0xffffffffu ? st.run_at : 0u;
  if (p.n_windows) p.n_windows[st.pair] = st.windows;
  if (p.cells) p.cells[st.pair] = st.cells;
}

template <int VW>
__device__ __forceinline__ void lane_begin(const AlignParams& p, uint32_t pair, LanePair<VW>& st,
                                           bool writer) {
  st.pair = pair;
  st.m = p.read_len[pair];
  st.n = p.ref_len[pair];
  st.read = p.reads + p.read_off[pair];
  st.ref = p.refs + p.ref_off[pair];
  const uint64_t c0 = p.cigar_off[pair];
  const uint64_t room = p.cigar_cap ? p.cigar_cap[pair] : p.cigar_off[pair + 1] - c0;
  st.out = p.cigar + c0;
  st.room = room > 0xffffffffull ? 0xffffffffu : static_cast<uint32_t>(room);
  st.cap = writer ? st.room : 0u;
  st.run_at = 0xffffffffu;
  st.run_op = st.run_len = 0u;
  st.cells = 0;
  st.pos_p = st.pos_t = st.edits = st.windows = 0;
  st.status = kPairOk;
  st.busy = true;
  if (p.ref_start) {  // free-start first window: begin where the locate step found
    const int32_t s0 = p.ref_start[pair];
    const int32_t dl = p.locate_d[pair];
    if (s0 < 0) {
      st.status = kPairExceedsK;
      lane_finish(p, st, writer);
      return;
    }
    st.pos_t = static_cast<uint32_t>(s0);
    if (dl >= 0) {
      const uint64_t span_end = static_cast<uint64_t>(p.start_span[pair]) + static_cast<uint64_t>(p.W);
      const uint64_t L = min(static_cast<uint64_t>(st.n), span_end);
      st.cells = L * static_cast<uint64_t>(dl + 1);
    }
  }
  if (st.m == 0) lane_finish(p, st, writer);  // empty read: nothing to align
}

// A pair's window state between turns of the sliced queue or serving steps
// (all zero: not started).
template <int VW>
__device__ __forceinline__ void lane_resume(const SlotState& s, LanePair<VW>& st) {
  st.pos_p = s.pos_p;
  st.pos_t = s.pos_t;
  st.edits = s.edits;
  st.windows = s.windows;
  st.cells = s.cells;
  st.run_at = s.runs - 1u;
  st.run_op = s.run_op;
  st.run_len = s.run_len;
}

template <int VW>
__device__ __forceinline__ void lane_save(const LanePair<VW>& st, SlotState& s) {
  s.pos_p = st.pos_p;
  s.pos_t = st.pos_t;
  s.edits = st.edits;
  s.windows = st.windows;
  s.cells = st.cells;
  s.runs = st.run_at + 1u;
  s.run_op = st.run_op;
  s.run_len = st.run_len;
}

}  // namespace ga
