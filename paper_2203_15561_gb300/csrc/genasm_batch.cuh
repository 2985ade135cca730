// The batched alignment kernel, the server's step kernel and the locate step
// as templates over the window width (VW 32-bit words per vector) and the
// traceback order; genasm_align.cu instantiates VW = 1 and 2 (windows of up
// to 32 and 64 bases), genasm_wide.cu VW = 3 and 4 (up to 96 and 128).
//
// Batched: a persistent grid of one-warp blocks; each lane pulls pairs from a
// device queue and aligns them one at a time, one window per round of its
// warp. With LPT the queue starts in longest-read-first order (a counting
// sort), so the lanes of a warp hold pairs of about the same length.
//
// Sliced form (slice > 0): the queue is a FIFO of pairs, and a lane runs a
// pair for a turn (`slice` windows, or a fraction of the pair's), saves its
// window state (positions, edit count, statistics, open CIGAR run) and puts it
// back at the tail. Every pair then moves forward at the same pace, and a batch
// whose pairs outnumber the resident lanes but not by a whole multiple does not
// end with a round in which a few lanes run alone.
//
// The FIFO is a bounded ring of 2n slots (n = pairs) with a sequence number
// per slot: position x lives in slot x % 2n; the slot holds position x's
// pair once its number is x + 1, and is free for position x + 2n once its
// number is x + 2n. A lane that wants a pair reserves the next head position
// with atomicAdd and takes the pair once that position is published; until
// then it stays idle while the other lanes of its warp go on (it checks
// again after each of their windows), and it stops once no pair is left
// unfinished. A lane that ends a turn claims the next tail position with
// atomicAdd; the slot it lands in held position y - 2n, which was published
// at least n pushes earlier and taken as soon as its reserver looked (at most
// n pairs are ever in the ring), so the slot is free; the lane writes the
// pair and publishes it. The wait for a free slot is bounded: should it run
// out, the lane keeps its pair for another turn and flags the launch, and the
// reserver of the lost position stops with the others at the end. Every pair
// not yet finished is held by a running lane or published in the ring. A
// warp whose lanes all wait for a pair also waits a bounded time only
// (behind a lost position published pairs could otherwise be left without a
// reserver); the pairs a run-out wait leaves unfinished keep the timed-out
// status that the ring's set-up kernel gives every pair.
#pragma once

#include <algorithm>
#include <cstdint>

#include <cuda_runtime.h>

#include "genasm.h"
#include "genasm_internal.h"
#include "genasm_lane.cuh"

namespace ga {

struct BatchArgs {
  uint32_t* queue;        // [0] hand-out counter (unsliced); ring: [1] head, [2] tail,
                          // [3] pairs not finished, [4] a warp's wait ran out,
                          // with `order`, what the lengths say: [5] turns pay, [6]
                          // lanes of a warp to use (0: all), [8..16] the split of
                          // the longest over the warps (see length_split; 0: none)
  const uint32_t* order;  // hand-out order (nullptr: index order)
  int cols;               // columns of a lane's table
  int lanes;              // lanes of a warp that take pairs
  uint32_t slice;         // windows per turn (0: a pair runs to its end)
  uint32_t turns;         // if not 0: turns only where they pay (queue[5]), each this fraction
                          // of its pair and `slice` windows at least
  uint32_t* ring;         // 2n ring slots: pair ids
  uint32_t* ring_seq;     // 2n: each slot's sequence number
  SlotState* state;       // per pair: saved window state (all zero: not started)
  uint32_t idle_polls;    // bound of a warp's wait for a published pair
  uint32_t push_polls;    // bound of a push's wait for its slot
};

constexpr uint32_t kNoPair = 0xffffffffu;

// The pair at reserved ring position x, or kNoPair while it is not published.
__device__ __forceinline__ uint32_t ring_take(const BatchArgs& a, uint32_t cap, uint32_t x) {
  volatile uint32_t* seq = a.ring_seq;
  volatile uint32_t* slot = a.ring;
  const uint32_t s = x % cap;
  if (seq[s] != x + 1u) return kNoPair;
  __threadfence();
  const uint32_t pair = slot[s];
  __threadfence();
  seq[s] = x + cap;  // free for position x + cap
  return pair;
}

// Puts a pair (its state already saved) at the ring's tail; false (the pair
// stays with its lane) only if the slot's wait ran out.
__device__ __forceinline__ bool ring_push(const BatchArgs& a, uint32_t cap, uint32_t pair) {
  volatile uint32_t* seq = a.ring_seq;
  volatile uint32_t* slot = a.ring;
  __threadfence();  // the saved state before the publication
  const uint32_t y = atomicAdd(a.queue + 2, 1u);
  const uint32_t s = y % cap;
  for (uint32_t polls = 0; seq[s] != y; ++polls) {
    if (polls >= a.push_polls) {
      atomicExch(a.queue + 4, 1u);
      return false;
    }
    __nanosleep(200);
  }
  slot[s] = pair;
  __threadfence();
  seq[s] = y + 1u;
  return true;
}

// The dynamic shared memory of a one-warp block, from its first multiple of
// the Eq masks' size on (their addresses are formed with OR).
template <class Shape>
__device__ __forceinline__ uint32_t lane_smem_base() {
  extern __shared__ __align__(1024) uint32_t lane_smem[];
  return (smem_addr(lane_smem) + Shape::kEqBytes - 1u) & ~(Shape::kEqBytes - 1u);
}
template <class Shape>
constexpr size_t lane_block_smem(int cols, bool any_order, bool staged) {
  return Shape::bytes(cols, any_order, staged) + (Shape::kEqBytes > 1024u ? 1024u : 0u);
}

// Hands `*counter`'s next values to the pairs of the lanes in `wants`, in lane
// order (the lanes of a pair want together).
template <class Shape>
__device__ __forceinline__ uint32_t take_next(uint32_t* counter, uint32_t wants, uint32_t lane) {
  const uint32_t pairs = wants & Shape::kLeaders;
  const int first = __ffs(pairs) - 1;
  uint32_t idx = 0;
  if (static_cast<int>(lane) == first) idx = atomicAdd(counter, __popc(pairs));
  return __shfl_sync(Shape::kMask, idx, first) + __popc(pairs & ((2u << lane) - 1u)) - 1u;
}

// Windows of a turn of a pair of m read bases.
__device__ __forceinline__ uint32_t turn_windows(const AlignParams& p, const BatchArgs& a, uint32_t m) {
  if (!a.turns) return a.slice;
  return max(a.slice, m / (static_cast<uint32_t>(p.W - p.O) * a.turns) + 1u);
}

template <int VW, int LP, int NL, bool kAny, bool kStaged>
__global__ void __launch_bounds__(LP * NL) align_batched_kernel(const AlignParams p, const BatchArgs a) {
  using Shape = LaneShape<VW, LP, NL>;
  constexpr uint32_t kMask = Shape::kMask;
  const uint32_t base = lane_smem_base<Shape>();
  const uint32_t lane = threadIdx.x;
  const uint32_t slot = lane / NL;
  const int leader = static_cast<int>(slot * NL);
  const bool writer = lane % NL == 0;
  const uint32_t slice = a.slice && (!a.turns || a.queue[5]) ? a.slice : 0u;
  uint32_t lanes = static_cast<uint32_t>(a.lanes);
  if (a.order && !slice && a.queue[6]) lanes = min(lanes, a.queue[6]);
  // The first pairs go round the warps lane by lane, so that the longest ones
  // (handed out first) are spread over all schedulers; then each lane takes the
  // next one when it is done.
  uint32_t deal = slot * gridDim.x + blockIdx.x, dealt = gridDim.x * lanes;
  if constexpr (kStaged && VW == 2) {
    if (a.order && !slice && a.queue[8 + kSplits - 1]) {
      // The long ones are split over the first warps, few lanes each; the others go
      // round the rest, all lanes.
      uint32_t warps = 0, given = 0, end = p.n_pairs;
      lanes = 0;
      for (int k = 0; k < kSplits; ++k) {
        const uint32_t upto = a.queue[8 + k], l = kSplitLanes(k), w = (upto - given + l - 1u) / l;
        if (lanes == 0 && blockIdx.x < warps + w) {
          lanes = l;
          deal = given + (blockIdx.x - warps) * l + slot;
          end = upto;
        }
        warps += w;
        given = upto;
      }
      dealt = given + (gridDim.x - warps) * 32u;
      if (lanes == 0) {
        lanes = 32;
        deal = given + slot * (gridDim.x - warps) + (blockIdx.x - warps);
      }
      if (deal >= end) deal = p.n_pairs;
    }
  }
  LanePair<VW> st{};
  bool drained = slot >= lanes;
  bool first = true;        // nothing handed out to this warp yet
  uint32_t budget = 0;
  // The ring position this lane has reserved. As without turns, the first pairs
  // go round the warps lane by lane.
  uint32_t resv = slot * gridDim.x + blockIdx.x;
  uint32_t idle = 0;        // consecutive polls of a warp with no pair to work on
  for (;;) {
    // Lanes without a pair take the next one from the queue.
    const bool want = !st.busy && !drained;
    const uint32_t wants = __ballot_sync(kMask, want);
    bool ended = false;  // a pair that finished at its start
    if (wants) {
      uint32_t pair = kNoPair;
      bool quit = false;
      if (slice) {
        if (want && writer) {
          if (resv == kNoPair) resv = atomicAdd(a.queue + 1, 1u);
          pair = ring_take(a, 2u * p.n_pairs, resv);
          if (pair != kNoPair) resv = kNoPair;
          else quit = *reinterpret_cast<volatile uint32_t*>(a.queue + 3) == 0u;  // all finished
        }
        if constexpr (NL > 1) {
          pair = __shfl_sync(kMask, pair, leader);
          quit = __shfl_sync(kMask, quit ? 1u : 0u, leader) != 0u;
        }
      } else {
        uint32_t idx = deal;
        if (!first) idx = p.n_pairs > dealt ? dealt + take_next<Shape>(a.queue, wants, lane) : p.n_pairs;
        if (want) {
          if (idx < p.n_pairs) pair = a.order ? a.order[idx] : idx;
          else quit = true;
        }
      }
      first = false;
      if (want) {
        if (pair != kNoPair) {
          lane_begin(p, pair, st, writer);
          ended = !st.busy;
          if (slice) {
            // Another SM may have saved this state: read it from L2, not L1.
            const SlotState* sp = a.state + pair;
            SlotState s;
            s.pos_p = __ldcg(&sp->pos_p);
            s.pos_t = __ldcg(&sp->pos_t);
            s.edits = __ldcg(&sp->edits);
            s.windows = __ldcg(&sp->windows);
            s.cells = __ldcg(reinterpret_cast<const unsigned long long*>(&sp->cells));
            s.runs = __ldcg(&sp->runs);
            s.run_op = __ldcg(&sp->run_op);
            s.run_len = __ldcg(&sp->run_len);
            if (s.windows > 0) lane_resume(s, st);  // a pair that had turns already
            budget = turn_windows(p, a, st.m);
          }
          if (st.busy) lane_fetch<VW, kStaged>(st, base);
        } else if (quit) {
          drained = true;
        }
      }
      __syncwarp(kMask);
      if (!__any_sync(kMask, st.busy)) {
        if (slice && __any_sync(kMask, ended)) {
          if (ended && writer) atomicSub(a.queue + 3, 1u);
          continue;
        }
        if (!__any_sync(kMask, !drained)) break;
        if (slice) {
          // Every lane of the warp waits for a pair: poll again shortly.
          __nanosleep(200);
          if (++idle >= a.idle_polls) {
            if (lane == 0) atomicExch(a.queue + 4, 1u);
            break;
          }
        }
        continue;
      }
      idle = 0;
    } else if (!__any_sync(kMask, st.busy)) {
      break;
    }
    // Windows until some lane's pair is done or its turn over (a lane that waits
    // for a pair looks again after each).
    bool done, turn;
    do {
      lane_window<VW, LP, NL, kAny, kStaged>(p, st, base, a.cols);
      done = st.busy && lane_done(st);
      turn = slice && st.busy && !done && --budget == 0;
    } while (!__any_sync(kMask, done || turn || (!st.busy && !drained)));
    if (done) lane_finish(p, st, writer);
    if (slice) {
      if ((done || ended) && writer) atomicSub(a.queue + 3, 1u);  // this pair is finished
      // End of a turn: the pair goes back to the queue's tail (or, if the ring
      // cannot take it now, stays for another turn).
      bool pushed = false;
      if (turn && writer) {
        lane_save(st, a.state[st.pair]);
        pushed = ring_push(a, 2u * p.n_pairs, st.pair);
      }
      if constexpr (NL > 1) pushed = __shfl_sync(kMask, pushed ? 1u : 0u, leader) != 0u;
      if (turn) {
        if (pushed) st.busy = false;
        else budget = turn_windows(p, a, st.m);
      }
    }
    __syncwarp(kMask);
  }
  if constexpr (kStaged) copies_wait();
}

// Serving step: resumable alignment. Every pair in the active list advances by
// at most `windows` windows; its window state is kept in device memory between
// steps, so pairs admitted at different times share one launch. The active list
// is read from, and the finished slots are written to, host memory mapped into
// the device: the warp that is last to finish writes their count and leaves the
// counters at zero for the next step, so that a step is this launch alone.
template <int VW>
__global__ void __launch_bounds__(32) align_step_kernel(const AlignParams p, const StepArgs a) {
  using Shape = LaneShape<VW, 32, 1>;
  constexpr uint32_t kMask = Shape::kMask;
  const uint32_t base = lane_smem_base<Shape>();
  const uint32_t lane = threadIdx.x;
  // Few pairs are spread over all warps.
  const uint32_t lanes = min(32u, (a.n_active + gridDim.x - 1) / gridDim.x);
  LanePair<VW> st{};
  bool drained = lane >= lanes;
  uint32_t slot = 0, budget = 0;
  for (;;) {
    const bool want = !st.busy && !drained;
    const uint32_t wants = __ballot_sync(kMask, want);
    bool finished = false;
    if (wants) {
      const uint32_t idx = take_next<Shape>(&a.counters[0], wants, lane);
      if (want) {
        if (idx < a.n_active) {
          slot = a.active[idx];
          lane_begin(p, slot, st, true);  // a fresh slot (all zero) starts here
          if (st.busy) {
            lane_resume(a.state[slot], st);
            lane_fetch<VW, false>(st, base);
          }
          budget = a.windows;
          finished = !st.busy;
        } else {
          drained = true;
        }
      }
      __syncwarp(kMask);
    }
    if (!__any_sync(kMask, st.busy || !drained || finished)) break;
    if (__any_sync(kMask, st.busy)) {
      bool done, turn;
      do {
        lane_window<VW, 32, 1, false, false>(p, st, base, a.cols);
        done = st.busy && lane_done(st);
        turn = st.busy && !done && --budget == 0;
      } while (!__any_sync(kMask, done || turn || finished));
      if (done) {
        lane_finish(p, st, true);
        finished = true;
      } else if (turn) {
        lane_save(st, a.state[slot]);
        st.busy = false;  // resumes at the next step
      }
    }
    if (finished) a.done[atomicAdd(&a.counters[1], 1u)] = slot;
    __syncwarp(kMask);
  }
  __threadfence_system();  // this warp's finished slots, before its arrival
  __syncwarp(kMask);
  if (lane == 0 && atomicAdd(&a.counters[2], 1u) == gridDim.x - 1) {
    __threadfence();
    *a.n_done = atomicExch(&a.counters[1], 0u);
    a.counters[0] = 0u;
    a.counters[2] = 0u;
  }
}

// ---------------------------------------------------------------------------
// Free-start first window: the locate step. For a pair with start span S > 0
// the first read window's pattern (wp = min(W, m) bases) is searched in the
// reference's first L = min(n, S + W) bases with the recurrence of the
// windows; every start column s = 0..min(S, L) is a candidate (s = L, the
// empty text, costs wp insertions) and the leftmost column with the fewest
// edits is where the alignment begins.
//
// 2^log_q lanes search a pair, each a range of start columns. A start's edits
// are at most wp, so its alignment spans at most 2 wp text bases: a lane whose
// recurrence begins 2 wp columns right of its range has every value of the
// range exactly. Within a lane the columns run right to left; the pattern's last
// row is counted at each word of start columns and followed through it by its
// horizontal differences; a column that does not cost more than the best one so
// far takes its place (ties go left). Words of other columns are the recurrence
// alone.
// ---------------------------------------------------------------------------

constexpr int kLocateWarps = 4;  // per block

struct LocateArgs {
  const uint32_t* start_span;
  int32_t* ref_start;
  int32_t* locate_d;
};

template <int VW>
__global__ void __launch_bounds__(32 * kLocateWarps)
    locate_kernel(const AlignParams p, const LocateArgs a, int log_q) {
  using Shape = LaneShape<VW, 32, 1>;
  // The Eq masks start at a multiple of their size (shared memory itself is
  // aligned to 1 KB at most).
  constexpr uint32_t kAlign = Shape::kEqBytes;
  __shared__ __align__(1024) uint32_t eqs[(kLocateWarps * kAlign + (VW >= 3 ? 1024u : 0u)) / 4];
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t eq_lane = ((smem_addr(eqs) + kAlign - 1u) & ~(kAlign - 1u)) +
                           (threadIdx.x >> 5) * kAlign + lane * Shape::kEqLane;
  const uint64_t gid = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const uint32_t q = 1u << log_q, part = lane & (q - 1u);
  const uint64_t pair = gid >> log_q;
  const bool valid = pair < p.n_pairs;
  uint32_t m = 0, n = 0, S = 0;
  if (valid) {
    m = p.read_len[pair];
    n = p.ref_len[pair];
    S = a.start_span[pair];
  }
  const bool go = valid && S > 0 && m > 0;
  const int wp = go ? static_cast<int>(min(m, static_cast<uint32_t>(p.W))) : 1;
  const uint64_t span_end = static_cast<uint64_t>(S) + static_cast<uint64_t>(p.W);
  const uint32_t L = go ? static_cast<uint32_t>(min(static_cast<uint64_t>(n), span_end)) : 0u;
  // The empty text (s = L) is a candidate when S reaches it: wp insertions.
  uint64_t best = ~0ull;
  if (go && S >= L && wp <= p.kmax) best = (static_cast<uint64_t>(wp) << 32) | L;
  // This lane's start columns [lo, hi) and the column its recurrence begins at.
  const uint32_t starts = go ? min(S == 0xffffffffu ? S : S + 1u, L) : 0u;
  const uint32_t per = (starts + q - 1u) >> log_q;
  const uint32_t lo = min(part * per, starts);
  const uint32_t hi = min(lo + per, starts);
  if (lo < hi) {
    uint32_t raw[2 * VW + 1], pw[2 * VW], PL[VW], PH[VW];
    const uint8_t* read = p.reads + p.read_off[pair];
    load_words<VW>(read, m, 0u, raw);
    align_bases<VW>(read, 0u, raw, pw);
    bit_planes<VW>(pw, PL, PH);
    store_eq<VW, 32, 1>(eq_lane, 0u, wp, PL, PH);
    const uint32_t x0 = static_cast<uint32_t>(min(static_cast<uint64_t>(L), static_cast<uint64_t>(hi) - 1u + 2u * wp));
    const uint8_t* ref = p.refs + p.ref_off[pair];
    const uintptr_t at = reinterpret_cast<uintptr_t>(ref);
    const uint32_t* words = reinterpret_cast<const uint32_t*>(at & ~static_cast<uintptr_t>(3));
    const uint32_t o = 4u * static_cast<uint32_t>(at & 3u);  // base 0's place in word 0
    uint32_t vp[VW], vn[VW], top[VW];
#pragma unroll
    for (int k = 0; k < VW; ++k) {
      vp[k] = ~0u;
      vn[k] = 0u;
      top[k] = (wp - 1) >> 5 == k ? 1u << ((wp - 1) & 31) : 0u;
    }
    const uint32_t top_at = static_cast<uint32_t>(wp - 1) & 31u;
    int found = 0x7fffffff;
    uint32_t pos = 0;
    const int64_t w0 = (static_cast<int64_t>(o) + lo) >> 4;
    int64_t w = (static_cast<int64_t>(o) + x0 - 1) >> 4;
    uint32_t tw = __ldg(words + w);
    uint32_t next = w > w0 ? __ldg(words + w - 1) : 0u;
    uint32_t e_hi[8][VW], e_lo[8][VW];
    load_eq8<VW>(eq_lane, tw, 8, e_hi);
    for (; w >= w0; --w) {
      const int64_t i0 = 16 * w - o;  // the word's first base
      load_eq8<VW>(eq_lane, tw, 0, e_lo);
      // Columns of the word at or past x0 keep the initial column.
      if (x0 - i0 < 16) {
        const int left = static_cast<int>(x0 - i0);
#pragma unroll
        for (int x = 0; x < 8; ++x) {
#pragma unroll
          for (int k = 0; k < VW; ++k) {
            e_lo[x][k] = x < left ? e_lo[x][k] : 0u;
            e_hi[x][k] = x + 8 < left ? e_hi[x][k] : 0u;
          }
        }
      }
      if (i0 >= hi) {  // no start column of this lane's in the word
#pragma unroll
        for (int x = 15; x >= 0; --x) {
          uint32_t d0[VW], hp[VW], hn[VW];
          column_step<VW>(x >= 8 ? e_hi[x & 7] : e_lo[x & 7], vp, vn, d0, hp, hn);
        }
      } else {
        // Start columns of the word: places from .. to - 1.
        const int to = hi - i0 < 16 ? static_cast<int>(static_cast<int64_t>(hi) - i0) : 16;
        const int from = i0 < lo ? static_cast<int>(lo - i0) : 0;
        int score = 0;
#pragma unroll
        for (int k = 0; k < VW; ++k) score += word_distance(wp, k, vp[k], vn[k]);
#pragma unroll
        for (int x = 15; x >= 0; --x) {
          uint32_t d0[VW], hp[VW], hn[VW];
          column_step<VW>(x >= 8 ? e_hi[x & 7] : e_lo[x & 7], vp, vn, d0, hp, hn);
          uint32_t up = 0, down = 0;
#pragma unroll
          for (int k = 0; k < VW; ++k) {
            up |= hp[k] & top[k];
            down |= hn[k] & top[k];
          }
          score += static_cast<int>(up >> top_at) - static_cast<int>(down >> top_at);
          const bool better = x < to && x >= from && score <= found;
          found = better ? score : found;
          pos = better ? static_cast<uint32_t>(i0 + x) : pos;
        }
      }
      tw = next;
      if (w > w0 + 1) next = __ldg(words + w - 2);
      load_eq8<VW>(eq_lane, tw, 8, e_hi);  // (past the last word: not used)
    }
    if (found <= p.kmax)
      best = min(best, (static_cast<uint64_t>(found) << 32) | pos);
  }
  __syncwarp();
  for (uint32_t s = q >> 1; s > 0; s >>= 1) best = min(best, __shfl_xor_sync(kFull, best, s));
  if (valid && part == 0) {
    if (!go) {
      a.ref_start[pair] = 0;
      a.locate_d[pair] = -1;
    } else if (best == ~0ull) {
      a.ref_start[pair] = -1;
      a.locate_d[pair] = -1;
    } else {
      a.ref_start[pair] = static_cast<int32_t>(best & 0xffffffffu);
      a.locate_d[pair] = static_cast<int32_t>(best >> 32);
    }
  }
}

// ---------------------------------------------------------------------------
// Launch shapes
// ---------------------------------------------------------------------------

// Opts the batched kernel in to a block's whole shared memory (whatever this
// launch takes of it: concurrent launches of other shapes need other sizes) and,
// unless warps_per_sm is null, reads the shape's resident warps per SM.
constexpr int kSharedOptIn = 227 * 1024;

template <int VW, int LP, int NL, bool kAny, bool kStaged>
cudaError_t lane_setup(int cols, int* warps_per_sm) {
  using Shape = LaneShape<VW, LP, NL>;
  const auto kernel = align_batched_kernel<VW, LP, NL, kAny, kStaged>;
  const cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSharedOptIn);
  if (e != cudaSuccess || !warps_per_sm) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(warps_per_sm, kernel, Shape::kThreads,
                                                       lane_block_smem<Shape>(cols, kAny, kStaged));
}

template <int VW, int LP, int NL>
cudaError_t lane_setup_order(const LanePlan& plan, int* warps_per_sm) {
  if constexpr (VW <= 2) {
    if (plan.staged)
      return plan.any_order ? lane_setup<VW, LP, NL, true, true>(plan.cols, warps_per_sm)
                            : lane_setup<VW, LP, NL, false, true>(plan.cols, warps_per_sm);
  }
  return plan.any_order ? lane_setup<VW, LP, NL, true, false>(plan.cols, warps_per_sm)
                        : lane_setup<VW, LP, NL, false, false>(plan.cols, warps_per_sm);
}

template <int VW, int LP, int NL, bool kAny, bool kStaged>
void lane_launch_as(const AlignParams& p, const LanePlan& plan, const BatchArgs& a, cudaStream_t s) {
  using Shape = LaneShape<VW, LP, NL>;
  align_batched_kernel<VW, LP, NL, kAny, kStaged>
      <<<plan.warps, Shape::kThreads, lane_block_smem<Shape>(plan.cols, kAny, kStaged), s>>>(p, a);
}

template <int VW, int LP, int NL>
void lane_launch(const AlignParams& p, const LanePlan& plan, const BatchArgs& a, cudaStream_t s) {
  if constexpr (VW <= 2) {
    if (plan.staged) {
      if (plan.any_order) lane_launch_as<VW, LP, NL, true, true>(p, plan, a, s);
      else lane_launch_as<VW, LP, NL, false, true>(p, plan, a, s);
      return;
    }
  }
  if (plan.any_order) lane_launch_as<VW, LP, NL, true, false>(p, plan, a, s);
  else lane_launch_as<VW, LP, NL, false, false>(p, plan, a, s);
}

template <int VW>
void locate_launch(const AlignParams& p, const LocateArgs& a, int log_q, cudaStream_t s) {
  const uint64_t threads = static_cast<uint64_t>(p.n_pairs) << log_q;
  const uint32_t per = 32u * kLocateWarps;
  locate_kernel<VW><<<static_cast<uint32_t>((threads + per - 1) / per), per, 0, s>>>(p, a, log_q);
}

// Windows of 65..128 bases (genasm_wide.cu).
cudaError_t wide_lane_setup(const LanePlan& plan, int* warps_per_sm);
void wide_lane_launch(const AlignParams& p, const LanePlan& plan, const BatchArgs& a, cudaStream_t s);
void wide_locate_launch(int vw, const AlignParams& p, const LocateArgs& a, int log_q, cudaStream_t s);

}  // namespace ga
