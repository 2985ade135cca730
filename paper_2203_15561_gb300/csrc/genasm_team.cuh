// A pair by a team of lanes: its next windows computed before it is known where
// they start (windows of up to 64 bases, default traceback order).
//
// The windows of a pair form a chain: each starts where the traceback of the one
// before stopped. A pair alone in its warp therefore costs the latency of a
// window (4,700 cycles of preparation, columns and traceback for a read against
// its place, 8,300 for sequences that do not match) times its windows, on one
// lane of 32. But the next start is not unknown, only uncertain: a window commits
// W - O bases of the read or of the text, whichever is used up first, and a few
// less of the other, as its insertions and deletions have it. So the lanes of a
// team each take one likely start of one of the next windows, all run their
// window to its end (columns, traceback, and CIGAR runs into shared memory), and
// then the team follows the chain through the results: from the first window,
// whose start is known, to the lane that guessed where it ended, and so on until
// nobody did. The results are those of the windows one after the other, exactly;
// a window that nobody guessed is the next round's first.
//
// Which starts: those that a model of the windows' indels holds most likely
// (genasm_team.cu), by what the pair has shown so far: a read of few errors, one
// of long-read errors, or sequences that do not belong together (their alignments
// fall behind on the text by some bases per window). Windows per round at 12%
// errors: 4.5 for 128 lanes, 2.8 for 32, 2.2 for 16, 1.8 for 8.
//
// A round of 128 lanes takes 8,350 cycles: 1,050 of preparation, 3,230 of columns
// (integer ALU, one warp per scheduler), 2,320 of traceback (the longest walk of
// the warp's lanes), 1,300 to follow the chain and write its runs; by 32 lanes
// 7,100, the chain 770. Calls of one 10 kb pair: 625 us with one lane, 277 (283
// with all warps at every window's runs). 16 requests of up to 64 mixed pairs at
// the server: 5.9 ms, 3.4.
#pragma once

#include <cstdint>

#include "genasm_internal.h"
#include "genasm_batch.cuh"

namespace ga {

// Shared memory of a block of NB warps: per warp the Eq masks, the tables of all
// columns and a window's runs of every lane; then what each lane found, and each
// team's table of its starts (32 places per lane).
template <int VW, int NB>
struct TeamShape {
  using Lane = LaneShape<VW, 32, 1>;
  static constexpr int kThreads = 32 * NB;
  static constexpr int kCols = 32 * VW;
  static constexpr uint32_t kRuns = 64u * VW;  // most runs of a window
  static constexpr uint32_t kTables =
      static_cast<uint32_t>((Lane::bytes(kCols, false, false) + Lane::kEqBytes - 1) / Lane::kEqBytes * Lane::kEqBytes);
  static constexpr uint32_t kWarp = kTables + kRuns * 128u;
  static_assert(kWarp % Lane::kEqBytes == 0, "every warp's Eq masks at a multiple of their size");
  static constexpr uint32_t kPosts = NB * kWarp;            // 32 bytes per thread
  static constexpr uint32_t kPlaces = kPosts + NB * 1024u;  // 32 bytes per thread
  static constexpr size_t kBytes = kPlaces + NB * 1024u;
};

// The runs of a window as its traceback finds them (see close_run): run k of a
// lane at `to` + 128 k.
struct WindowRuns {
  uint32_t run_at, run_op, run_len, edits, to;
};
__device__ __forceinline__ void sts32_if(bool when, uint32_t a, uint32_t x) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %0, 0;\n\t@p st.shared.u32 [%1], %2;\n\t}" ::"r"(
                   static_cast<uint32_t>(when)),
               "r"(a), "r"(x)
               : "memory");
}
__device__ __forceinline__ void sts8(uint32_t a, uint32_t x) {
  asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(x) : "memory");
}
__device__ __forceinline__ uint32_t lds8(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void close_run(WindowRuns& st, bool when) {
  sts32_if(when && st.run_at != 0xffffffffu, st.to + st.run_at * 128u, st.run_len << 4 | st.run_op);
  st.run_at += when ? 1u : 0u;
  st.run_len = when ? 0u : st.run_len;
}

// A lane's place in its team, and its starts: windows ahead (bits 0..3), and the
// bases that the read (4..9) and the text (10..15) are short of as many times
// W - O.
struct TeamLane {
  uint32_t rank, size, first;  // first: the team's first thread of the block
  uint32_t places, bits_p, bits_t;  // the table of its starts: 2^bits_p rows of 2^bits_t
  uint32_t start[kTeamKinds];
};
template <int NB>
__device__ __forceinline__ TeamLane team_lane(int log_size, const TeamStarts& s, uint32_t places) {
  TeamLane t;
  t.size = NB > 1 ? 32u * NB : 1u << log_size;
  t.rank = threadIdx.x & (t.size - 1u);
  t.first = threadIdx.x - t.rank;
  const uint32_t bits = 5u + (NB > 1 ? 7u : static_cast<uint32_t>(log_size));
  t.bits_t = bits / 2u;
  t.bits_p = bits - t.bits_t;
  t.places = places + t.first * 32u;
  // Places that no start has taken yet name the team's first thread. (Never one of
  // another team: its pair's starts may have the same numbers.)
  for (uint32_t k = 0; k < 8u; ++k) sts32(places + threadIdx.x * 32u + 4u * k, t.first * 0x01010101u);
#pragma unroll
  for (int k = 0; k < kTeamKinds; ++k) t.start[k] = s.start[k][t.rank];
  return t;
}

// A team's pair (the same in all its lanes), and what its windows since it was
// taken up have shown: their number, their edits and by how many bases the text
// has moved on less than the read.
template <int VW>
struct TeamPair {
  LanePair<VW> st;
  uint32_t seen, edits;
  int32_t behind;
};

template <int NB>
__device__ __forceinline__ void team_sync() {
  if constexpr (NB > 1) __syncthreads();
  else __syncwarp();
}

// The place of the start that lies on_p and on_t bases on: some windows ahead,
// the starts differ by few bases in the read and in the diagonal, so that hardly
// two share a place (if they do, one is lost).
__device__ __forceinline__ uint32_t team_place(const TeamLane& me, uint32_t on_p, uint32_t on_t) {
  return me.places + ((on_p & ((1u << me.bits_p) - 1u)) << me.bits_t | ((on_p - on_t) & ((1u << me.bits_t) - 1u)));
}

// Brings the 128 bytes of a sequence from the sector after that of base `pos` on
// into L1 (lane k of four, a sector each), for the windows to come.
__device__ __forceinline__ void team_ahead(const uint8_t* seq, uint32_t len, uint32_t pos, uint32_t k) {
  const uint32_t at = (pos >> 2) + 32u * (k + 1u);
  if (at < len >> 2) {
    uint32_t v;
    asm volatile("ld.global.nc.u8 %0, [%1];" : "=r"(v) : "l"(seq + at));
    (void)v;
  }
}

// The windows of the team's pair from its position on, one to many of them, at
// most `budget`.
template <int VW, int NB>
__device__ __forceinline__ void team_windows(const AlignParams& p, TeamPair<VW>& tp, const TeamLane& me,
                                             uint32_t base, uint32_t budget) {
  using Team = TeamShape<VW, NB>;
  using Shape = typename Team::Lane;
  LanePair<VW>& st = tp.st;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp_base = base + (NB > 1 ? (threadIdx.x >> 5) * Team::kWarp : 0u);
  const uint32_t eq_lane = warp_base + lane * Shape::kEqLane;
  const uint32_t tab_lane = warp_base + Shape::kEqBytes + lane * Shape::kPairBytes;
  const uint32_t runs_lane = warp_base + Team::kTables + lane * 4u;
  const uint32_t posts = base + Team::kPosts;
  const uint32_t commit = static_cast<uint32_t>(p.W - p.O);

  // This lane's window.
  const bool few = tp.seen >= 4u && tp.edits <= tp.seen;
  const bool strange = tp.seen >= 4u && tp.behind > 0 && 12u * static_cast<uint32_t>(tp.behind) > tp.seen * commit;
  const uint32_t start = few ? me.start[kTeamFew] : strange ? me.start[kTeamStrange] : me.start[kTeamLong];
  const uint32_t ahead = start & 15u;
  uint32_t short_t = start >> 10;
  if (strange && me.rank > 0) {
    const uint32_t lag = __float2uint_rn(static_cast<float>(ahead * static_cast<uint32_t>(tp.behind)) *
                                         __frcp_rn(static_cast<float>(tp.seen)));
    short_t = lag + short_t > 32u ? lag + short_t - 32u : 0u;
  }
  const uint32_t on_p = ahead * commit - ((start >> 4) & 63u), on_t = ahead * commit - short_t;
  const uint32_t at_p = st.pos_p + on_p, at_t = st.pos_t + on_t;
  // (bases on, as signed numbers: a start before the pair's position is none)
  const bool ga = st.busy && static_cast<int32_t>(on_p) >= 0 && static_cast<int32_t>(on_t) >= 0 &&
                  on_p < st.m - st.pos_p && on_t <= st.n - st.pos_t;
  int wp = 1, wt = 0;
  if (ga) {
    wp = static_cast<int>(min(static_cast<uint32_t>(p.W), st.m - at_p));
    wt = static_cast<int>(min(static_cast<uint32_t>(p.W), st.n - at_t));
  }
  const bool last = !ga || at_p + static_cast<uint32_t>(wp) == st.m;
  Walk<VW, 32, 1> w;
  uint32_t tw[2 * VW];
  {
    uint32_t raw_p[2 * VW + 1], raw_t[2 * VW + 1], pw[2 * VW];
    const uint32_t from_p = ga ? at_p : 0u, from_t = ga ? at_t : 0u;
    load_words<VW>(st.read, ga ? st.m : 0u, from_p, raw_p);
    load_words<VW>(st.ref, ga ? st.n : 0u, from_t, raw_t);
    if (st.busy && me.rank < 8u) {
      if (me.rank < 4u) team_ahead(st.read, st.m, st.pos_p, me.rank);
      else team_ahead(st.ref, st.n, st.pos_t, me.rank - 4u);
    }
    if (ga) sts8(team_place(me, on_p, on_t), threadIdx.x);
    align_bases<VW>(st.read, from_p, raw_p, pw);
    align_bases<VW>(st.ref, from_t, raw_t, tw);
    bit_planes<VW>(pw, w.pl, w.ph);
    bit_planes<VW>(tw, w.tl, w.th);
  }
  store_eq<VW, 32, 1>(eq_lane, 0u, wp, w.pl, w.ph);
  w.plane_lane = 0u;
  w.tab0 = tab_lane;
  w.hp0 = 0u;
  w.top = static_cast<uint32_t>(wp) - 1u;
  const int ncols16 = (p.W + 15) >> 4;
  const bool inner = !last && static_cast<int>(commit) <= wt;
  uint32_t goal = !ga ? 0u : last ? static_cast<uint32_t>(wp) : commit;
  const uint32_t text = inner ? commit : static_cast<uint32_t>(wt);
  const bool mask = __any_sync(0xffffffffu, ga && (wt < 16 * ncols16 || !inner));
  const int end = mask ? Team::kCols : static_cast<int>(commit);
  const int dmin = mask ? window_columns<VW, 32, true, false>(wp, wt, ncols16, tw, eq_lane, tab_lane, 0u, 0, end)
                        : window_columns<VW, 32, false, false>(wp, wt, ncols16, tw, eq_lane, tab_lane, 0u, 0, end);
  const bool fails = dmin > p.kmax;
  if (fails) goal = 0u;
  uint32_t cp = 0, ct = 0;
  WindowRuns rw{0xffffffffu, 0u, 0u, 0u, runs_lane};
  LateOps late{0u, 0u};
  while (cp < goal && ct < text) {
    walk_step<VW, 32, 1>(w, rw, cp, ct, goal, text, late);
    walk_step<VW, 32, 1>(w, rw, cp, ct, goal, text, late);
  }
  book_ops(rw, late);
  if (cp < goal && !inner) {  // the text is used up
    close_run(rw, rw.run_op != kOpIns);
    rw.run_op = kOpIns;
    rw.run_len += goal - cp;
    rw.edits += goal - cp;
    cp = goal;
  }
  // What it found: its start, where it ended, cells, edits and whether it failed,
  // its runs and the first and the last of them, and who guessed its end.
  const uint32_t runs = rw.run_at + 1u, open = rw.run_len << 4 | rw.run_op;
  const uint32_t run0 = runs > 1u ? lds32(runs_lane) : open;
  const uint32_t post = posts + threadIdx.x * 32u;
  const uint32_t end_p = at_p + cp, end_t = at_t + ct;
  sts64(post + 24u, ga ? at_p : 0xffffffffu, at_t);
  team_sync<NB>();
  const uint32_t next = lds8(team_place(me, end_p - st.pos_p, end_t - st.pos_t));
  const uint2 its = lds64(posts + next * 32u + 24u);
  // (bit 24: nobody; 25: it failed)
  const uint32_t found = static_cast<uint32_t>(wt) * static_cast<uint32_t>(dmin + 1) | rw.edits << 13 |
                         (its.x != end_p || its.y != end_t ? 1u << 24 : 0u) | (fails ? 1u << 25 : 0u);
  sts128(post, end_p, end_t, found, next | runs << 8);
  sts64(post + 16u, run0, open);
  team_sync<NB>();

  // The chain of windows through the results, by every lane of the team alike;
  // the next one's are read before this one's are used. The warps of a block take
  // turns at writing the windows' runs; `entry` is this lane's run of the window.
  const uint32_t place = NB > 1 ? lane : me.rank, places = NB > 1 ? 32u : me.size;
  const uint32_t lists = base + Team::kTables + place * 128u;
  const auto list_of = [&](uint32_t t) {
    return lists + (NB > 1 ? (t >> 5) * Team::kWarp + (t & 31u) * 4u : t * 4u);
  };
  bool live = st.busy;
  uint32_t turn = NB > 1 ? threadIdx.x >> 5 : 0u;
  uint4 a = lds128(posts + me.first * 32u);
  uint2 b = lds64(posts + me.first * 32u + 16u);
  uint32_t entry = lds32(list_of(me.first)), cur = me.first;
  while (live) {
    const uint32_t then = a.w & 255u;
    const uint4 a1 = lds128(posts + then * 32u);
    const uint2 b1 = lds64(posts + then * 32u + 16u);
    const uint32_t entry1 = lds32(list_of(then));
    // Its runs join the pair's, the first one perhaps the open run. (A window that
    // failed has none, any other one at least.)
    const uint32_t r = a.w >> 8;
    const bool joins = (b.x & 15u) == st.run_op;
    const uint32_t add = joins ? st.run_len : 0u;
    const uint32_t to = st.run_at + (joins ? 0u : 1u);
    if (NB == 1 || (turn++ & (NB - 1u)) == 0u) {
      stg32_if(!joins && place == 0u && r > 0u && st.run_at < st.room, st.out + st.run_at,
               st.run_len << 4 | st.run_op);
      stg32_if(place + 1u < r && to + place < st.room, st.out + to + place,
               entry + (place == 0u ? add << 4 : 0u));
      for (uint32_t i = place + places; i + 1u < r; i += places)
        stg32_if(to + i < st.room, st.out + to + i, lds32(list_of(cur) + (i - place) * 128u));
    }
    if (a.z >> 25) {
      st.status = kPairExceedsK;
      break;
    }
    st.run_at = to + r - 1u;
    st.run_op = b.y & 15u;
    st.run_len = (b.y >> 4) + (r == 1u ? add : 0u);
    if (static_cast<int32_t>(st.run_at) >= 0 && st.run_at > st.room) {
      st.status = kPairCigarFull;
      break;
    }
    const uint32_t edits = (a.z >> 13) & 255u;
    ++st.windows;
    st.cells += a.z & 8191u;
    st.edits += edits;
    tp.edits += edits;
    ++tp.seen;
    tp.behind += static_cast<int32_t>((a.x - st.pos_p) - (a.y - st.pos_t));
    st.pos_p = a.x;
    st.pos_t = a.y;
    live = st.pos_p < st.m && --budget > 0u && (a.z >> 24) == 0u;
    a = a1;
    b = b1;
    entry = entry1;
    cur = then;
  }
  team_sync<NB>();  // the results have been read
}

template <int VW>
__device__ __forceinline__ void team_begin(const AlignParams& p, uint32_t pair, TeamPair<VW>& tp, bool writer) {
  lane_begin(p, pair, tp.st, writer);
  tp.seen = tp.edits = 0u;
  tp.behind = 0;
}

// Batches of no more pairs than resident teams (a grid of one wave): the pairs
// go round the blocks.
template <int VW, int NB>
__global__ void __launch_bounds__(32 * NB)
    align_team_kernel(const AlignParams p, const uint32_t* order, int log_size, const __grid_constant__ TeamStarts starts) {
  const uint32_t base = lane_smem_base<typename TeamShape<VW, NB>::Lane>();
  const TeamLane me = team_lane<NB>(log_size, starts, base + TeamShape<VW, NB>::kPlaces);
  team_sync<NB>();
  TeamPair<VW> tp{};
  const uint32_t teams = gridDim.x * (32u * NB / me.size);
  uint32_t idx = me.first / me.size * gridDim.x + blockIdx.x;
  for (;;) {
    bool more = false;
    if (!tp.st.busy && idx < p.n_pairs) {
      team_begin(p, order ? order[idx] : idx, tp, me.rank == 0u);
      idx = p.n_pairs - idx > teams ? idx + teams : p.n_pairs;
      more = true;
    }
    if (!__any_sync(0xffffffffu, tp.st.busy)) {
      if (!__any_sync(0xffffffffu, more)) break;
      continue;
    }
    team_windows<VW, NB>(p, tp, me, base, 0xffffffffu);
    if (tp.st.busy && lane_done(tp.st)) lane_finish(p, tp.st, me.rank == 0u);
  }
}

// Serving step (see align_step_kernel) by teams.
template <int VW, int NB>
__global__ void __launch_bounds__(32 * NB)
    step_team_kernel(const AlignParams p, const StepArgs a, int log_size, const __grid_constant__ TeamStarts starts) {
  const uint32_t base = lane_smem_base<typename TeamShape<VW, NB>::Lane>();
  const TeamLane me = team_lane<NB>(log_size, starts, base + TeamShape<VW, NB>::kPlaces);
  team_sync<NB>();
  TeamPair<VW> tp{};
  const uint32_t teams = gridDim.x * (32u * NB / me.size);
  uint32_t idx = me.first / me.size * gridDim.x + blockIdx.x;
  uint32_t slot = 0, until = 0;
  for (;;) {
    bool more = false, finished = false;
    if (!tp.st.busy && idx < a.n_active) {
      slot = a.active[idx];
      idx = a.n_active - idx > teams ? idx + teams : a.n_active;
      more = true;
      team_begin(p, slot, tp, me.rank == 0u);  // a fresh slot (all zero) starts here
      if (tp.st.busy) lane_resume(a.state[slot], tp.st);
      until = tp.st.windows + a.windows;
      finished = !tp.st.busy;
    }
    if (__any_sync(0xffffffffu, tp.st.busy)) {
      team_windows<VW, NB>(p, tp, me, base, until - tp.st.windows);
      if (tp.st.busy) {
        if (lane_done(tp.st)) {
          lane_finish(p, tp.st, me.rank == 0u);
          finished = true;
        } else if (tp.st.windows == until) {
          if (me.rank == 0u) lane_save(tp.st, a.state[slot]);
          tp.st.busy = false;  // resumes at the next step
        }
      }
    } else if (!__any_sync(0xffffffffu, more)) {
      break;
    }
    if (finished && me.rank == 0u) a.done[atomicAdd(&a.counters[1], 1u)] = slot;
  }
  __threadfence_system();  // this block's finished slots, before its arrival
  team_sync<NB>();
  if (threadIdx.x == 0 && atomicAdd(&a.counters[2], 1u) == gridDim.x - 1) {
    __threadfence();
    *a.n_done = atomicExch(&a.counters[1], 0u);
    a.counters[2] = 0u;
  }
}

}  // namespace ga
