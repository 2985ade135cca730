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

namespace ga {

// Shared memory of a warp. Eq: four masks of VW words per lane. Table: per
// stored column and word {D0, VP'}, then (orders other than the default) HP.
// Planes (VW >= 3): the low and high code bits of the window's read and
// reference bases, VW words and a zero each.
template <int VW>
struct LaneShape {
  static constexpr int kBases = 32 * VW;
  static constexpr uint32_t kEqLane = VW == 1 ? 4u : VW == 2 ? 8u : 16u;  // bytes per lane and mask
  static constexpr uint32_t kEqBytes = 4u * 32u * kEqLane;
  static constexpr uint32_t kPlaneBytes = VW >= 3 ? 4u * (VW + 1) * 128u : 0u;
  static constexpr uint32_t kColBytes = VW * 256u;   // {D0, VP'} of one column, 32 lanes
  static constexpr uint32_t kHpBytes = VW * 128u;    // HP of one column, 32 lanes
};

__host__ __device__ constexpr uint32_t lane_smem_bytes(int VW, int cols, bool any_order) {
  const uint32_t eq = 4u * 32u * (VW == 1 ? 4u : VW == 2 ? 8u : 16u);
  const uint32_t planes = VW >= 3 ? 4u * (VW + 1) * 128u : 0u;
  return eq + planes + static_cast<uint32_t>(cols) * VW * (any_order ? 384u : 256u);
}

// A pair in the hands of a lane.
struct LanePair {
  const uint8_t* read;
  const uint8_t* ref;
  uint32_t* out;      // its CIGAR runs
  uint64_t cells;
  uint32_t cap;       // room for runs
  uint32_t runs;      // runs closed so far (those past cap are counted, not stored)
  uint32_t cur;       // the open run (length << 4 | op), 0: none
  uint32_t pair, m, n, pos_p, pos_t, edits, windows;
  int32_t status;
  bool busy;
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

// The 32 * VW bases at `pos` of a packed sequence of `len` bases (16 per word;
// past the end of the sequence: anything). Only aligned words that hold a
// base of the sequence are read.
template <int VW>
__device__ __forceinline__ void load_bases(const uint8_t* seq, uint32_t len, uint32_t pos,
                                           uint32_t (&w)[2 * VW]) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(seq) + (pos >> 2);
  const uint32_t* wa = reinterpret_cast<const uint32_t*>(a & ~static_cast<uintptr_t>(3));
  const uint32_t o = 8u * static_cast<uint32_t>(a & 3u) + 2u * (pos & 3u);
  const uint32_t lim = o + 2u * min(len > pos ? len - pos : 0u, 32u * VW);  // first bit past the window
  uint32_t x[2 * VW + 1];
#pragma unroll
  for (int k = 0; k <= 2 * VW; ++k) x[k] = 32u * k < lim ? __ldg(wa + k) : 0u;
#pragma unroll
  for (int k = 0; k < 2 * VW; ++k) w[k] = __funnelshift_r(x[k], x[k + 1], o);
}

// Low and high code bits of the bases in `w`: bit u of L / H is base u's.
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
    L[k] = __byte_perm(u[0], u[1], 0x6420);
    H[k] = __byte_perm(u[0], u[1], 0x7531);
  }
}

// Eq masks (bit j set iff P[wp-1-j] is the base) from the pattern's planes,
// into the lane's Eq words. Bits at and above wp: anything.
template <int VW>
__device__ __forceinline__ void store_eq(uint32_t eq_lane, int wp, const uint32_t (&L)[VW],
                                         const uint32_t (&H)[VW]) {
  // Reversed planes: bit j is base 32*VW-1-j's; then down by 32*VW - wp bits.
  uint32_t l[VW], h[VW];
  const uint32_t sh = static_cast<uint32_t>(32 * VW - wp);
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    l[k] = __brev(L[VW - 1 - k]);
    h[k] = __brev(H[VW - 1 - k]);
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
  constexpr uint32_t kRow = 32u * LaneShape<VW>::kEqLane;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    uint32_t e[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k)
      e[k] = (c & 1 ? l[k] : ~l[k]) & (c & 2 ? h[k] : ~h[k]);
    const uint32_t a = eq_lane + c * kRow;
    if constexpr (VW == 1) {
      sts32(a, e[0]);
    } else {
      sts64(a, e[0], e[1]);
      if constexpr (VW == 3) sts32(a + 8, e[2]);
      if constexpr (VW == 4) sts64(a + 8, e[VW - 2], e[VW - 1]);
    }
  }
}

// Address of the Eq masks of base x of a word of text bases.
template <int VW>
__device__ __forceinline__ uint32_t eq_at(uint32_t eq_lane, uint32_t tw, int x) {
  constexpr uint32_t kRow = 32u * LaneShape<VW>::kEqLane;  // a power of two, 128..512
  constexpr int kLog = VW == 1 ? 7 : VW == 2 ? 8 : 9;
  const int sh = 2 * x - kLog;
  const uint32_t c = sh >= 0 ? tw >> sh : tw << -sh;
  return eq_lane | (c & (3u * kRow));
}

// The Eq masks of bases x0 + 7 .. x0 of a word of text bases.
template <int VW>
__device__ __forceinline__ void load_eq8(uint32_t eq_lane, uint32_t tw, int x0,
                                         uint32_t (&e)[8][VW]) {
#pragma unroll
  for (int x = 7; x >= 0; --x) load_eq<VW>(eq_at<VW>(eq_lane, tw, x0 + x), e[x]);
}

// Eight columns, right to left from column c0 + 7, c0 of the window; their
// table entries go to `row` (column c0's) when `keep` is set.
template <int VW, bool kMask, bool kHp>
__device__ __forceinline__ void eight_columns(const uint32_t (&e)[8][VW], int left, bool keep,
                                              uint32_t row, uint32_t hrow, uint32_t (&vp)[VW],
                                              uint32_t (&vn)[VW]) {
#pragma unroll
  for (int x = 7; x >= 0; --x) {
    uint32_t eq[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) eq[k] = kMask && x >= left ? 0u : e[x][k];
    uint32_t d0[VW], hp[VW], hn[VW];
    column_step<VW>(eq, vp, vn, d0, hp, hn);
    if (keep) {
#pragma unroll
      for (int k = 0; k < VW; ++k) {
        sts64(row + x * LaneShape<VW>::kColBytes + k * 256, d0[k], vp[k]);
        if constexpr (kHp) sts32(hrow + x * LaneShape<VW>::kHpBytes + k * 128, hp[k]);
      }
    }
  }
}

// The columns of a window, right to left from column 16 * ncols16 - 1: the
// table entries of columns [cb, cb + cols) (multiples of 8) go to `tab_lane`.
// With kMask, columns at and past wt leave the initial column as it is (no
// base matches there: D(wt, j) = j + 1 repeats). Returns D(0, wp-1). The Eq
// masks are loaded eight columns ahead, before the stores of the columns in
// between: the recurrence itself never waits for shared memory.
template <int VW, bool kMask, bool kHp>
__device__ __forceinline__ int window_columns(int wp, int wt, int ncols16, uint32_t (&tw)[2 * VW],
                                              uint32_t eq_lane, uint32_t tab_lane, uint32_t hp_lane,
                                              int cb, int cols) {
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
  for (int b = ncols16 - 1; b >= 0; --b) {
    const int c0 = 16 * b - cb;  // the block's first column in the table
    const uint32_t row = tab_lane + static_cast<uint32_t>(c0) * LaneShape<VW>::kColBytes;
    const uint32_t hrow = hp_lane + static_cast<uint32_t>(c0) * LaneShape<VW>::kHpBytes;
    load_eq8<VW>(eq_lane, tw[2 * VW - 1], 0, lo);
    eight_columns<VW, kMask, kHp>(hi, wt - 16 * b - 8,
                                  static_cast<unsigned>(c0 + 8) < static_cast<unsigned>(cols),
                                  row + 8 * LaneShape<VW>::kColBytes,
                                  hrow + 8 * LaneShape<VW>::kHpBytes, vp, vn);
#pragma unroll
    for (int k = 2 * VW - 1; k > 0; --k) tw[k] = tw[k - 1];
    load_eq8<VW>(eq_lane, tw[2 * VW - 1], 8, hi);  // (past the last block: not used)
    eight_columns<VW, kMask, kHp>(lo, wt - 16 * b,
                                  static_cast<unsigned>(c0) < static_cast<unsigned>(cols), row,
                                  hrow, vp, vn);
  }
  int d = 0;
#pragma unroll
  for (int k = 0; k < VW; ++k) {
    const int bits = wp - 32 * k;
    const uint32_t mask = bits >= 32 ? ~0u : bits > 0 ? (1u << bits) - 1u : 0u;
    d += __popc(vp[k] & mask) - __popc(vn[k] & mask);
  }
  return d;
}

// Closes the open run of a pair. Runs past the capacity are counted only: the
// window's end turns the count into the pair's status.
__device__ __forceinline__ void emit_run(LanePair& st) {
  if (st.cur) {
    if (st.runs < st.cap) st.out[st.runs] = st.cur;
    ++st.runs;
  }
}
__device__ __forceinline__ void append_run(LanePair& st, uint32_t op, uint32_t len) {
  if ((st.cur & 15u) == op) {
    st.cur += len << 4;
  } else {
    emit_run(st);
    st.cur = len << 4 | op;
  }
}

// The 32 base bits from position c < 32 * VW on of a plane of VW words.
template <int VW>
__device__ __forceinline__ uint32_t plane_at(const uint32_t (&w)[VW], uint32_t plane_lane, int which,
                                             uint32_t c) {
  if constexpr (VW == 1) {
    return w[0] >> (c & 31u);
  } else if constexpr (VW == 2) {
    return static_cast<uint32_t>(((static_cast<uint64_t>(w[1]) << 32) | w[0]) >> (c & 63u));
  } else {
    const uint32_t a = plane_lane + which * (VW + 1) * 128u + min(c >> 5, VW - 1u) * 128u;
    return __funnelshift_r(lds32(a), lds32(a + 128u), c);
  }
}

// One window of the lane's pair (the window chain of a pair is serial: each
// window starts where the previous traceback stopped). Lanes without a pair
// come along with ga false. kAny: traceback orders other than M > S > I > D.
//
// The table holds `cols` columns (a multiple of 8); a traceback that walks
// past them has the columns computed again with the next `cols` stored.
template <int VW, bool kAny>
__device__ __forceinline__ void lane_window(const AlignParams& p, LanePair& st, uint32_t base,
                                            int cols) {
  using Shape = LaneShape<VW>;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t eq_lane = base + lane * Shape::kEqLane;
  const uint32_t plane_lane = base + Shape::kEqBytes + lane * 4u;
  const uint32_t tab_base = base + Shape::kEqBytes + Shape::kPlaneBytes;
  const uint32_t tab_lane = tab_base + lane * 8u;
  const uint32_t hp_lane = tab_base + static_cast<uint32_t>(cols) * Shape::kColBytes + lane * 4u;
  const bool ga = st.busy;
  const int commit = p.W - p.O;
  int wp = 1, wt = 0;
  bool last = true;
  uint32_t PL[VW], PH[VW], TL[VW], TH[VW], tw[2 * VW];
#pragma unroll
  for (int k = 0; k < 2 * VW; ++k) tw[k] = 0u;
#pragma unroll
  for (int k = 0; k < VW; ++k) PL[k] = PH[k] = 0u;
  if (ga) {
    wp = static_cast<int>(min(static_cast<uint32_t>(p.W), st.m - st.pos_p));
    wt = static_cast<int>(min(static_cast<uint32_t>(p.W), st.n - st.pos_t));
    last = st.pos_p + static_cast<uint32_t>(wp) == st.m;
    uint32_t pw[2 * VW];
    load_bases<VW>(st.read, st.m, st.pos_p, pw);
    load_bases<VW>(st.ref, st.n, st.pos_t, tw);
    bit_planes<VW>(pw, PL, PH);
  }
  store_eq<VW>(eq_lane, wp, PL, PH);
  bit_planes<VW>(tw, TL, TH);
  if constexpr (VW >= 3) {
#pragma unroll
    for (int k = 0; k <= VW; ++k) {
      const uint32_t a = plane_lane + k * 128u;
      sts32(a, k < VW ? PL[k < VW ? k : 0] : 0u);
      sts32(a + (VW + 1) * 128u, k < VW ? PH[k < VW ? k : 0] : 0u);
      sts32(a + 2u * (VW + 1) * 128u, k < VW ? TL[k < VW ? k : 0] : 0u);
      sts32(a + 3u * (VW + 1) * 128u, k < VW ? TH[k < VW ? k : 0] : 0u);
    }
  }
  const int ncols16 = (p.W + 15) >> 4;
  // A window that stops W - O bases in, before its text can run out, ends when
  // either count gets there; others end with their pattern bases (the text
  // used up: only insertions are left).
  const bool inner = !last && commit <= wt;
  int rp = last ? wp : commit;              // pattern bases left
  int rt = inner ? commit : wt;             // text bases left
  uint32_t cp = 0, ct = 0;
  int dmin = -1;
  bool run = ga;
  bool exceeds = false;
  for (int cb = 0;; cb += cols) {
    uint32_t t2[2 * VW];
#pragma unroll
    for (int k = 0; k < 2 * VW; ++k) t2[k] = tw[k];
    __syncwarp();
    const bool mask = __any_sync(kFull, ga && wt < 16 * ncols16);
    const int d = mask ? window_columns<VW, true, kAny>(wp, wt, ncols16, t2, eq_lane, tab_lane,
                                                        hp_lane, cb, cols)
                       : window_columns<VW, false, kAny>(wp, wt, ncols16, t2, eq_lane, tab_lane,
                                                         hp_lane, cb, cols);
    if (cb == 0 && ga) {
      dmin = d;
      exceeds = dmin > p.kmax;
      run = !exceeds;
    }
    const uint32_t ct_end = static_cast<uint32_t>(cb + cols);  // columns stored so far
    while (run && (ct < ct_end || rt == 0)) {
      if constexpr (!kAny) {
        // The matches ahead on this diagonal (32 at a time), then one edit.
        const uint32_t mm = (plane_at<VW>(PL, plane_lane, 0, cp) ^ plane_at<VW>(TL, plane_lane, 2, ct)) |
                            (plane_at<VW>(PH, plane_lane, 1, cp) ^ plane_at<VW>(TH, plane_lane, 3, ct));
        const int L = min(min(__clz(__brev(mm)), static_cast<int>(ct_end - ct)), min(rp, rt));
        cp += L;
        ct += L;
        rp -= L;
        rt -= L;
        if (L > 0) append_run(st, kOpMatch, L);
        if (rp == 0 || (rt == 0 && inner)) {
          run = false;
        } else if (rt == 0) {
          append_run(st, kOpIns, rp);
          st.edits += rp;
          cp += rp;
          run = false;
        } else if (ct < ct_end && L < 32) {
          const uint32_t j = static_cast<uint32_t>(wp) - 1u - cp;
          const uint2 e = lds64(tab_lane + ((ct - cb) * VW + (j >> 5)) * 256u);
          const uint32_t bit = 1u << (j & 31u);
          const bool s = (e.x & bit) == 0u;
          const bool del = !s && (e.y & bit) == 0u;
          const bool ins = !s && !del;
          append_run(st, s ? kOpSubst : ins ? kOpIns : kOpDel, 1u);
          ++st.edits;
          cp += del ? 0 : 1;
          rp -= del ? 0 : 1;
          ct += ins ? 0 : 1;
          rt -= ins ? 0 : 1;
        }
      } else {
        if (rp == 0 || (rt == 0 && inner)) {
          run = false;
        } else if (rt == 0) {
          append_run(st, kOpIns, rp);
          st.edits += rp;
          cp += rp;
          run = false;
        } else {
          const uint32_t j = static_cast<uint32_t>(wp) - 1u - cp;
          const uint32_t mm = (plane_at<VW>(PL, plane_lane, 0, cp) ^ plane_at<VW>(TL, plane_lane, 2, ct)) |
                              (plane_at<VW>(PH, plane_lane, 1, cp) ^ plane_at<VW>(TH, plane_lane, 3, ct));
          const uint32_t at = (ct - cb) * VW + (j >> 5);
          const uint2 e = lds64(tab_lane + at * 256u);
          const uint32_t h = lds32(hp_lane + at * 128u);
          const uint32_t bit = 1u << (j & 31u);
          const uint32_t can = ((mm & 1u) == 0u ? 1u << kTbM : 0u) | ((e.x & bit) == 0u ? 1u << kTbS : 0u) |
                               ((e.y & bit) != 0u ? 1u << kTbI : 0u) | ((h & bit) != 0u ? 1u << kTbD : 0u);
          const uint32_t code = static_cast<uint32_t>(p.tb_table >> (4 * can)) & 15u;
          append_run(st, (kTbOps >> (4u * code)) & 15u, 1u);
          st.edits += code != kTbM ? 1u : 0u;
          cp += code != kTbD ? 1 : 0;
          rp -= code != kTbD ? 1 : 0;
          ct += code != kTbI ? 1 : 0;
          rt -= code != kTbI ? 1 : 0;
        }
      }
    }
    __syncwarp();
    if (!__any_sync(kFull, run)) break;
  }
  if (ga) {
    if (exceeds) {
      st.status = kPairExceedsK;
    } else if (st.runs > st.cap) {
      st.status = kPairCigarFull;
    } else {
      ++st.windows;
      st.cells += static_cast<uint64_t>(wt) * static_cast<uint64_t>(dmin + 1);
      st.pos_p += cp;
      st.pos_t += ct;
    }
  }
}

__device__ __forceinline__ void lane_finish(const AlignParams& p, LanePair& st) {
  if (st.status == kPairOk) {
    emit_run(st);
    st.cur = 0u;
    if (st.runs > st.cap) st.status = kPairCigarFull;
  }
  const bool ok = st.status == kPairOk;
  p.dist[st.pair] = ok ? static_cast<int32_t>(st.edits) : -1;
  p.status[st.pair] = st.status;
  p.ref_consumed[st.pair] = ok ? static_cast<int32_t>(st.pos_t) : -1;
  if (p.ref_start && !ok) p.ref_start[st.pair] = -1;
  p.n_runs[st.pair] = ok ? st.runs : 0u;
  if (p.n_windows) p.n_windows[st.pair] = st.windows;
  if (p.cells) p.cells[st.pair] = st.cells;
  st.busy = false;
}

__device__ __forceinline__ void lane_begin(const AlignParams& p, uint32_t pair, LanePair& st) {
  st.pair = pair;
  st.m = p.read_len[pair];
  st.n = p.ref_len[pair];
  st.read = p.reads + p.read_off[pair];
  st.ref = p.refs + p.ref_off[pair];
  const uint64_t c0 = p.cigar_off[pair];
  const uint64_t room = p.cigar_cap ? p.cigar_cap[pair] : p.cigar_off[pair + 1] - c0;
  st.out = p.cigar + c0;
  st.cap = room > 0xffffffffull ? 0xffffffffu : static_cast<uint32_t>(room);
  st.runs = st.cur = 0u;
  st.cells = 0;
  st.pos_p = st.pos_t = st.edits = st.windows = 0;
  st.status = kPairOk;
  st.busy = true;
  if (p.ref_start) {  // free-start first window: begin where the locate step found
    const int32_t s0 = p.ref_start[pair];
    const int32_t dl = p.locate_d[pair];
    if (s0 < 0) {
      st.status = kPairExceedsK;
      lane_finish(p, st);
      return;
    }
    st.pos_t = static_cast<uint32_t>(s0);
    if (dl >= 0) {
      const uint64_t span_end = static_cast<uint64_t>(p.start_span[pair]) + static_cast<uint64_t>(p.W);
      const uint64_t L = min(static_cast<uint64_t>(st.n), span_end);
      st.cells = L * static_cast<uint64_t>(dl + 1);
    }
  }
  if (st.m == 0) lane_finish(p, st);  // empty read: nothing to align
}

// A pair's window state between turns of the sliced queue or serving steps.
__device__ __forceinline__ void lane_resume(const SlotState& s, LanePair& st) {
  st.pos_p = s.pos_p;
  st.pos_t = s.pos_t;
  st.edits = s.edits;
  st.windows = s.windows;
  st.cells = s.cells;
  st.runs = s.runs;
  st.cur = s.run_len ? s.run_len << 4 | s.run_op : 0u;
}

__device__ __forceinline__ void lane_save(const LanePair& st, SlotState& s) {
  s.pos_p = st.pos_p;
  s.pos_t = st.pos_t;
  s.edits = st.edits;
  s.windows = st.windows;
  s.cells = st.cells;
  s.runs = st.runs;
  s.run_op = st.cur & 15u;
  s.run_len = st.cur >> 4;
}

}  // namespace ga
