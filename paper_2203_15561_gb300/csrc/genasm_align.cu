// The batched alignment: pair order, ring set-up, launch shapes and launches
// (the kernels are in genasm_batch.cuh), and the server's step.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

#include "genasm.h"
#include "genasm_batch.cuh"
#include "genasm_internal.h"

namespace ga {

// Default bounds of the two waits (ga_set_queue_wait_limits changes them):
// polls of a warp whose lanes all wait for a pair (about 0.2 microseconds
// each): seconds, far beyond any legitimate wait (the rest of the longest
// pair); past it the warp stops and flags the launch. Polls of a push waiting
// for its slot: a fifth of a second at most.
constexpr uint32_t kRingPolls = 25u * 1000u * 1000u;
constexpr uint32_t kPushPolls = 1000u * 1000u;

// Counting sort of pairs by read length, longest first (LPT hand-out).
__device__ __forceinline__ uint32_t lpt_bucket(uint32_t read_len) {
  // 64-base buckets up to 65,535 bases; longer reads share the top bucket.
  const uint32_t b = read_len >> 6;
  return kLptBuckets - 1u - min(b, static_cast<uint32_t>(kLptBuckets - 1));
}

// Adds 1 to h[b] for every lane with `in` set and returns the value before this
// lane's. Lanes of a warp with the same bucket add together (reads of one length
// all fall into one bucket).
__device__ __forceinline__ uint32_t count_bucket(uint32_t* h, uint32_t b, bool in) {
  const uint32_t same = __match_any_sync(kFull, in ? b : 0xffffffffu);
  const uint32_t lane = threadIdx.x & 31u;
  const int first = __ffs(same) - 1;
  uint32_t at = 0;
  if (in && static_cast<int>(lane) == first) at = atomicAdd(&h[b], __popc(same));
  return __shfl_sync(kFull, at, first) + __popc(same & ((1u << lane) - 1u));
}

// Exclusive scan of kLptBuckets counts in shared memory, a thread each; s: one
// word per warp.
__device__ __forceinline__ uint32_t scan_buckets(uint32_t v, uint32_t* s) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, x, o);
    if (lane >= static_cast<uint32_t>(o)) x += y;
  }
  if (lane == 31u) s[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = s[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, w, o);
      if (lane >= static_cast<uint32_t>(o)) w += y;
    }
    s[lane] = w;
  }
  __syncthreads();
  return (warp ? s[warp - 1] : 0u) + x - v;
}

// What the pairs' lengths say about the launch, from the buckets' counts and
// starts in the order (a thread each; longest first):
//
// facts[0], whether the sliced queue pays: only when the pair that nine in ten
// are at least as long as has four fifths of the longest one's bases. Pairs of
// one length end in a round of few lanes without turns; of mixed lengths, the
// short ones at the end of the order fill the lanes up as the long ones finish,
// and turns cost more than they give (30,011 pairs of 2-20 kb: 2.32 ms with
// turns, 1.88 without; 20,000 of 100 bases-50 kb: 5.8 and 4.9). Not always: 138,929
// pairs of 2-20 kb anchored in a flank, in index order, take 10.1 ms with turns of 64
// windows and 17.3 longest first without, which the lengths do not show; the
// autotuner finds that.
//
// facts[1], the lanes per warp that finish all pairs by the time the longest one
// takes, and a quarter more: where a few long pairs decide, fewer lanes share
// their warps and their windows are shorter (the walk lasts as long as the
// warp's longest).
//
// facts[2], whether the order is to be that of the indexes: with a `choice`, an
// autotuned order and autotuned turns are taken if the lengths are of their kind,
// and facts[0] says whether turns are.
__device__ __forceinline__ void length_facts(uint32_t count, uint32_t start, uint32_t n, uint32_t warps,
                                             uint32_t choice, uint32_t* facts) {
  __shared__ uint32_t longest, ninth;
  __shared__ unsigned long long total;
  const uint32_t len = kLptBuckets - 1u - threadIdx.x;  // in 64 bases
  const uint32_t at = n - n / 10u - 1u;                 // the place of that pair
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  if (count && start == 0u) longest = len;
  if (count && start <= at && at < start + count) ninth = len;
  unsigned long long mine = static_cast<unsigned long long>(count) * (len + 1u);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(kFull, mine, o);
  if ((threadIdx.x & 31u) == 0u && mine) atomicAdd(&total, mine);
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool alike = 5u * (ninth + 1u) >= 4u * (longest + 1u);
    const bool tuned = choice && alike == ((choice & kChoiceAlike) != 0u);
    bool turns = alike && (!choice || (choice & kChoiceAutomatic));
    if (tuned && (choice & (kChoiceTurns | kChoiceNoTurns))) turns = (choice & kChoiceTurns) != 0u;
    const bool index = tuned && (choice & kChoiceIndex);
    facts[0] = turns ? 1u : 0u;
    const unsigned long long lanes = 5ull * total / (4ull * warps * (longest + 1u)) + 1ull;
    facts[1] = index ? 0u : lanes < 32ull ? static_cast<uint32_t>(lanes) : 32u;
    facts[2] = index ? 1u : 0u;
  }
}

// facts[3..11], where a few long pairs decide: how the first pairs of the order are
// split over the warps, pairs of about one length to a warp. A lane of a warp with
// l busy lanes takes about 2.33 + 0.47 log2(l) us per window (W = 64; the longest of
// l walks), so with a time t for the whole batch a pair of `len` may share its warp
// with as many lanes as let len * cost(l) stay within t. Of 32 times between the
// longest pair alone and in a full warp, the shortest whose warps suffice, all
// other pairs in full warps. facts[3 + s]: the pairs that get at most
// kSplitLanes(s) lanes. (The cost is fitted at W = 64, O = 24 and used for all W of 33
// to 64; only speed depends on it.) Only for vectors of two words and one warp per scheduler
// (the one-word kernel lost 2% at 5,000 equal pairs). Alignment with the same
// lanes in all warps, and split: 10,000 pairs of 2-20 kb 1.56 ms, 1.32; 5,000 of
// 100 bases-20 kb at W = 48 1.65, 1.47; 20,000 of 100 bases-50 kb 4.52, 4.26 (a long
// pair whose windows lose its path decides there).
__device__ __forceinline__ float lane_cost(float lanes) { return 2.33f + 0.47f * __log2f(lanes); }

__device__ __forceinline__ void length_split(uint32_t count, uint32_t start, uint32_t n, uint32_t warps,
                                             uint32_t* s, uint32_t* facts) {
  __shared__ uint32_t longer[kLptBuckets + 1], mass[kLptBuckets + 1];  // in buckets before x
  const uint32_t x = threadIdx.x;
  const uint32_t m = count * (kLptBuckets - x);
  longer[x] = start;
  mass[x] = scan_buckets(m, s);
  if (x == kLptBuckets - 1u) {
    longer[kLptBuckets] = n;
    mass[kLptBuckets] = mass[x] + m;
  }
  __syncthreads();
  if (x >= 32u || facts[0] || facts[2]) return;
  uint32_t top = 0;  // the longest pair's bucket
  for (uint32_t b = kLptBuckets / 2; b; b >>= 1)
    if (longer[top + b] == 0u) top += b;
  const float longest = static_cast<float>(kLptBuckets - top), all = lane_cost(32.0f);
  const float t = longest * (lane_cost(1.0f) + (all - lane_cost(1.0f)) * static_cast<float>(x) / 31.0f);
  uint32_t used = 0, at = kLptBuckets, given = 0;
  uint32_t upto[kSplits];
#pragma unroll
  for (int k = 0; k < kSplits; ++k) {
    const uint32_t more = k + 1 < kSplits ? kSplitLanes(k + 1) : 32u;
    const uint32_t len = static_cast<uint32_t>(t / lane_cost(static_cast<float>(more)));  // may have `more` lanes
    at = kLptBuckets - min(len, static_cast<uint32_t>(kLptBuckets));
    upto[k] = longer[at];
    used += (upto[k] - given + kSplitLanes(k) - 1u) / kSplitLanes(k);
    given = upto[k];
  }
  const float rest = static_cast<float>(mass[kLptBuckets] - mass[at]) * all * 1.05f;
  const bool fits = used < warps && rest <= t * 32.0f * static_cast<float>(warps - used);
  const uint32_t able = __ballot_sync(kFull, fits);
  // Against the same number of lanes in all warps.
  const float even = max(longest, static_cast<float>(mass[kLptBuckets]) / static_cast<float>(warps * facts[1])) *
                     lane_cost(static_cast<float>(facts[1]));
  if (able && x == static_cast<uint32_t>(__ffs(able)) - 1u && t < 0.95f * even) {
#pragma unroll
    for (int k = 0; k < kSplits; ++k) facts[3 + k] = upto[k];
  }
}

// The whole order of a batch of up to kLptOneBlock pairs by one block, which also
// zeroes the queue's counters.
constexpr uint32_t kLptOneBlock = 16384;

__global__ void __launch_bounds__(kLptBuckets)
    lpt_block_kernel(const uint32_t* __restrict__ read_len, uint32_t n, uint32_t warps, bool split,
                     uint32_t choice, uint32_t* queue, uint32_t* __restrict__ order) {
  __shared__ uint32_t h[kLptBuckets];
  __shared__ uint32_t s[32];
  const uint32_t x = threadIdx.x;
  if (x < 64u) queue[x] = 0u;
  h[x] = 0u;
  __syncthreads();
  const uint32_t rounds = (n + kLptBuckets - 1) / kLptBuckets;
  constexpr uint32_t kRounds = kLptOneBlock / kLptBuckets;
  uint32_t bucket[kRounds];  // all loads in flight at once
#pragma unroll
  for (uint32_t r = 0; r < kRounds; ++r) {
    const uint32_t q = r * kLptBuckets + x;
    bucket[r] = q < n ? lpt_bucket(read_len[q]) : 0u;
  }
#pragma unroll
  for (uint32_t r = 0; r < kRounds; ++r)
    if (r < rounds) count_bucket(h, bucket[r], r * kLptBuckets + x < n);
  __syncthreads();
  const uint32_t start = scan_buckets(h[x], s);
  length_facts(h[x], start, n, warps, choice, queue + 5);
  __syncthreads();
  const bool index = queue[7] != 0u;
  if (split) length_split(h[x], start, n, warps, s, queue + 5);
  h[x] = start;
  __syncthreads();
#pragma unroll
  for (uint32_t r = 0; r < kRounds; ++r) {
    if (r < rounds) {
      const uint32_t q = r * kLptBuckets + x;
      const uint32_t at = count_bucket(h, bucket[r], q < n);
      if (q < n) order[index ? q : at] = q;
    }
  }
}

// Larger batches in three launches. Each block counts its own pairs in shared
// memory and reserves their places in the order with one addition per bucket.
constexpr uint32_t kLptPairs = 8 * kLptBuckets;  // pairs per block

__device__ __forceinline__ void lpt_count(const uint32_t* __restrict__ read_len, uint32_t n, uint32_t* h) {
  const uint64_t q0 = static_cast<uint64_t>(blockIdx.x) * kLptPairs + threadIdx.x;
  h[threadIdx.x] = 0u;
  __syncthreads();
#pragma unroll
  for (uint32_t r = 0; r < kLptPairs / kLptBuckets; ++r) {
    const uint64_t q = q0 + r * kLptBuckets;
    count_bucket(h, q < n ? lpt_bucket(read_len[q]) : 0u, q < n);
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kLptBuckets)
    lpt_histogram_kernel(const uint32_t* __restrict__ read_len, uint32_t n, uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[kLptBuckets];
  lpt_count(read_len, n, h);
  if (h[threadIdx.x]) atomicAdd(&hist[threadIdx.x], h[threadIdx.x]);
}

// Exclusive scan of the bucket counts in place (one block of kLptBuckets threads).
__global__ void __launch_bounds__(kLptBuckets) lpt_scan_kernel(uint32_t* hist, uint32_t n, uint32_t warps,
                                                                bool split, uint32_t choice, uint32_t* facts) {
  __shared__ uint32_t s[32];
  const uint32_t count = hist[threadIdx.x];
  const uint32_t start = scan_buckets(count, s);
  if (facts) length_facts(count, start, n, warps, choice, facts);
  __syncthreads();
  if (facts && split) length_split(count, start, n, warps, s, facts);
  hist[threadIdx.x] = start;
}

__global__ void __launch_bounds__(kLptBuckets)
    lpt_scatter_kernel(const uint32_t* __restrict__ read_len, uint32_t n, const uint32_t* __restrict__ facts,
                       uint32_t* __restrict__ cursor, uint32_t* __restrict__ order) {
  __shared__ uint32_t h[kLptBuckets];
  const bool index = facts && facts[2] != 0u;
  lpt_count(read_len, n, h);
  const uint32_t mine = h[threadIdx.x];
  const uint32_t start = mine ? atomicAdd(&cursor[threadIdx.x], mine) : 0u;
  __syncthreads();
  h[threadIdx.x] = start;
  __syncthreads();
  const uint64_t q0 = static_cast<uint64_t>(blockIdx.x) * kLptPairs + threadIdx.x;
#pragma unroll
  for (uint32_t r = 0; r < kLptPairs / kLptBuckets; ++r) {
    const uint64_t q = q0 + r * kLptBuckets;
    const uint32_t at = count_bucket(h, q < n ? lpt_bucket(read_len[q]) : 0u, q < n);
    if (q < n) order[index ? q : at] = static_cast<uint32_t>(q);
  }
}

cudaError_t launch_lpt_order(const uint32_t* read_len, uint32_t n, uint32_t* hist, uint32_t* order,
                             uint32_t warps, bool split, uint32_t choice, uint32_t* facts, cudaStream_t s) {
  const uint32_t blocks =
      static_cast<uint32_t>((static_cast<uint64_t>(n) + kLptPairs - 1) / kLptPairs);
  lpt_histogram_kernel<<<blocks, kLptBuckets, 0, s>>>(read_len, n, hist);
  lpt_scan_kernel<<<1, kLptBuckets, 0, s>>>(hist, n, warps, split, choice, facts);
  lpt_scatter_kernel<<<blocks, kLptBuckets, 0, s>>>(read_len, n, facts, hist, order);
  count_launches(3);
  return cudaGetLastError();
}

// The ring of the sliced queue (2n slots) starts with every pair: slot x < n
// holds hand-out position x (the LPT order, or pair x), published with
// sequence number x + 1; slots n..2n-1 are free for positions n..2n-1. Every
// pair starts as timed out (distance and reference end -1, no runs): a pair
// that finishes overwrites it, and one left in the ring when a bounded wait
// ran out keeps it.
// The positions 0 .. dealt-1 are reserved by the lanes before they start (see
// the kernel), so the head begins past them.
__global__ void ring_init_kernel(uint32_t n, uint32_t dealt, const uint32_t* __restrict__ order,
                                 uint32_t* __restrict__ ring, uint32_t* __restrict__ seq,
                                 uint32_t* __restrict__ queue, SlotState* __restrict__ state,
                                 int32_t* __restrict__ status,
                                 int32_t* __restrict__ dist, int32_t* __restrict__ ref_consumed,
                                 uint32_t* __restrict__ n_runs) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    queue[1] = dealt;
    if (!order) queue[5] = 1u;  // no order, nothing known of the lengths: take turns
    queue[2] = n;  // tail: the ring starts with every pair
    queue[3] = n;  // pairs not finished
  }
  for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < 2u * n; x += gridDim.x * blockDim.x) {
    if (x < n) {
      ring[x] = order ? order[x] : x;
      state[x] = SlotState{};
      status[x] = kPairTimedOut;
      dist[x] = -1;
      ref_consumed[x] = -1;
      n_runs[x] = 0u;
    }
    seq[x] = x < n ? x + 1u : x;
  }
}

namespace {
std::atomic<uint32_t> g_idle_polls{kRingPolls};
std::atomic<uint32_t> g_push_polls{kPushPolls};
}  // namespace

void set_queue_wait_limits(uint32_t idle_polls, uint32_t push_polls) {
  g_idle_polls.store(idle_polls ? idle_polls : kRingPolls, std::memory_order_relaxed);
  g_push_polls.store(push_polls ? push_polls : kPushPolls, std::memory_order_relaxed);
}

// ---------------------------------------------------------------------------
// Tunings
// ---------------------------------------------------------------------------

// The launch shapes a tuning may name. They are checked as they always were
// (a saved tuning stays valid, a wrong one is still an error); the batched
// kernel runs one lane per pair and takes `lpt` and `slice_windows` from it.
bool batch_variant_exists(int G, int max_registers) {
  if (max_registers == 0 || max_registers == 255) return G == 4 || G == 8 || G == 16 || G == 32;
  return G == 8 && (max_registers == 168 || max_registers == 128);
}

namespace {

bool banded(int O) { return O >= 16; }
int shape_stride(int G, int ncols) {
  const int q = G == 32 ? 2 : 4;
  return (ncols + q - 1) / q * q;
}
int shape_entries(int G, int W, int O, int rows) {
  const int ncols = W - O + 1;
  return banded(O) ? std::max((rows * shape_stride(G, ncols) + 1) / 2, kMaxW)
                   : rows * table_stride(ncols) + kMaxW;
}

}  // namespace

cudaError_t resolve_tuning(int W, int O, int k, const ga_tuning* t, int mode, ga_tuning* out,
                           int* made_for) {
  ga_tuning d{8, 8, 39, 1, 0, 0};
  *made_for = kMadeForAny;
  stored_tuning(W, O, k, &d, made_for, mode);  // chosen by an autotuner or set by ga_tuning_set
  if (t && *made_for != kMadeForAny) d.lpt = 1;  // (an autotuned order goes with autotuned turns)
  if (t) *made_for = kMadeForAny;
  // (a stored tuning without its own shape has the library's)
  const int rows = d.table_rows;
  int entries = shape_entries(d.lanes_per_pair, W, O, rows);
  ga_tuning r = d;
  r.lpt = d.lpt >= 0 ? 1 : -1;
  if (t) {
    if (t->lanes_per_pair) r.lanes_per_pair = t->lanes_per_pair;
    if (t->pairs_per_block) r.pairs_per_block = t->pairs_per_block;
    if (t->table_rows) {
      r.table_rows = t->table_rows;
      entries = shape_entries(r.lanes_per_pair, W, O, t->table_rows);
    }
    if (t->lpt) r.lpt = t->lpt > 0 ? 1 : -1;
    r.max_registers = t->max_registers;
    r.slice_windows = t->slice_windows;
    if (t->table_rows < 0 || r.slice_windows < -1) return cudaErrorInvalidValue;
  }
  const int G = r.lanes_per_pair, ppb = r.pairs_per_block;
  if (!batch_variant_exists(G, r.max_registers) || ppb < 1 || ppb * G > 256 || (ppb * G) % 32 != 0)
    return cudaErrorInvalidValue;
  entries = std::max(kMaxStride + kMaxW, std::min(entries, kMaxRows * kMaxStride + kMaxW)) & ~1;
  int dev = 0, smem_optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  if (static_cast<size_t>(ppb) * (256 + 8ull * entries) > static_cast<size_t>(smem_optin))
    return cudaErrorInvalidValue;
  *out = r;
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Launch shapes
// ---------------------------------------------------------------------------

namespace {

int vw_for(int W) { return (W + 31) / 32; }
int up8(int x) { return (x + 7) / 8 * 8; }

cudaError_t setup_for(const LanePlan& plan, int* warps_per_sm) {
  if (plan.vw == 1) return lane_setup_order<1, 32, 1>(plan, warps_per_sm);
  if (plan.vw == 2) return lane_setup_order<2, 32, 1>(plan, warps_per_sm);
  return wide_lane_setup(plan, warps_per_sm);
}

}  // namespace

namespace {

// What a launch asks the driver about the device, asked once: SMs, and the
// resident warps of each launch shape (a call of every shape costs a few
// microseconds, a tenth of a small batch). Shapes differ by width, pairs per
// warp, order, staging and table columns (multiples of 8 up to 128).
struct DeviceFacts {
  int sms = 0;
  int8_t warps[4][3][2][2][17] = {};  // 0: not asked yet, else warps per SM + 1
};
constexpr int kMaxDevices = 64;
std::mutex g_facts_mutex;
DeviceFacts g_facts[kMaxDevices];

cudaError_t device_sms(int* dev, int* sms) {
  cudaError_t e = cudaGetDevice(dev);
  if (e != cudaSuccess) return e;
  if (*dev < 0 || *dev >= kMaxDevices)
    return cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, *dev);
  std::lock_guard<std::mutex> lock(g_facts_mutex);
  DeviceFacts& f = g_facts[*dev];
  if (f.sms == 0) e = cudaDeviceGetAttribute(&f.sms, cudaDevAttrMultiProcessorCount, *dev);
  *sms = f.sms;
  return e;
}

cudaError_t shape_warps(int dev, const LanePlan& plan, int* warps) {
  if (dev < 0 || dev >= kMaxDevices) return setup_for(plan, warps);
  std::lock_guard<std::mutex> lock(g_facts_mutex);
  int8_t& w = g_facts[dev].warps[plan.vw - 1][plan.lp == 32 ? 0 : plan.lp == 16 ? 1 : 2][plan.any_order]
                                [plan.staged][plan.cols / 8];
  cudaError_t e = cudaSuccess;
  if (w == 0) {
    e = setup_for(plan, warps);
    if (e == cudaSuccess) w = static_cast<int8_t>(*warps + 1);
  }
  *warps = w - 1;
  return e;
}

}  // namespace

cudaError_t lane_plan(const AlignParams& p, int slice_windows, bool asked, bool lpt, int made_for,
                      LanePlan* plan) {
  int dev = 0, sms = 0;
  cudaError_t e = device_sms(&dev, &sms);
  if (e != cudaSuccess) return e;
  plan->vw = vw_for(p.W);
  plan->any_order = p.tb_table != tb_table(kTbOrderDefault);
  const bool tuned = made_for != kMadeForAny;
  plan->lpt = lpt || tuned;  // (the ordering finds out whether a tuning is for these lengths)
  plan->choice = 0;
  const uint64_t n = std::max<uint32_t>(p.n_pairs, 1);
  const uint64_t scheds = 4ull * sms;
  const int all = up8(p.W), inner = up8(p.W - p.O);
  int per_sm = 0;
  // Few pairs: a team of lanes each, in one wave (no order needed; turns only if
  // the call itself asks for them: a stored tuning was chosen for some other batch,
  // and one pair of 10 kb takes 840 us with its turns, 295 by a team).
  const bool turns_asked = slice_windows > 0 && asked;
  plan->team = plan->vw <= 2 && !plan->any_order && !turns_asked ? team_size(n, sms) : 0;
  if (plan->team) {
    plan->lp = 32;
    plan->cols = 32 * plan->vw;
    plan->staged = false;
    plan->slice = plan->turns = 0;
    plan->lanes = std::max(1, 32 / plan->team);
    plan->warps = static_cast<int>(std::min<uint64_t>(plan->team > 32 ? sms : scheds, n));
    return cudaSuccess;
  }
  // Windows of 65 bases and more: four lanes per pair while one warp per
  // scheduler holds every pair (2,001 pairs of 10 kb at W = 128: 0.79 ms against
  // 1.16 with one lane each). At W <= 64 two lanes per pair gained nothing (3,330
  // cycles for a window's columns against 3,280).
  plan->staged = false;
  if (plan->vw >= 3 && n <= 8 * scheds) {
    plan->lp = 8;
    plan->cols = all;
    if ((e = shape_warps(dev, *plan, &per_sm)) != cudaSuccess) return e;
    per_sm = std::min(per_sm, 4);
  } else {
    // One lane per pair. Tables of every column a window can walk, else of the W
    // - O columns of windows that are not a pair's last; warps of 32 pairs, else
    // of 16: the first that leaves each of an SM's four schedulers as many warps
    // as the pairs can use, else the one with most. That is one warp until the
    // pairs fill two rounds of it, then two: with every lane busy two warps per
    // scheduler take 1.49 times as long per window as one (38,912 pairs of 2 kb
    // 312 us, 19,456 pairs 209), but with pairs for half the lanes 1.9 times
    // (10,000 pairs of 10 kb: 2.05 ms against 1.10).
    const int want = n > 64 * scheds ? 8 : 4;
    LanePlan best = *plan, t = *plan;
    t.staged = plan->vw <= 2 && want == 4 && n > scheds;
    for (int lp : {32, 16}) {
      if (lp == 16 && plan->vw < 3) break;
      for (int cols : {all, std::max(inner, std::min(all, 48)), inner}) {
        if (per_sm >= want) break;
        t.lp = lp;
        t.cols = cols;
        int ps = 0;
        if ((e = shape_warps(dev, t, &ps)) != cudaSuccess) return e;
        ps = ps >= 8 ? 8 : std::min(ps, 4);
        if (ps <= per_sm) continue;
        per_sm = ps;
        best = t;
      }
      if (per_sm >= 4) break;
    }
    *plan = best;
    per_sm = std::min(per_sm, want);
  }
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // (an attribute of the function in this context: set for every launch)
  if ((e = setup_for(*plan, nullptr)) != cudaSuccess) return e;
  const uint64_t warps = std::min<uint64_t>(static_cast<uint64_t>(sms) * per_sm, n);
  plan->warps = static_cast<int>(warps);
  plan->lanes = static_cast<int>(std::min<uint64_t>(plan->lp, (n + warps - 1) / warps));
  // The sliced queue: turns of the call's choice, else of 64 windows or a quarter
  // of the pair when the pairs outnumber the resident lanes less than 16 times over
  // (more pairs than that leave a tail of under a sixteenth of a round) and are of
  // about one length, which the ordering finds out on the device (length_facts).
  // Stored turns are taken where the pairs outnumber the lanes and are of about one
  // length (stored turns of 64, and without them: 10,000 pairs of 10 kb 1.18 ms,
  // 0.97; 20,000 of 100 bases-50 kb 5.72, 4.26), autotuned ones and an autotuned
  // order where the pairs outnumber the lanes and are of the kind they were made for
  // (138,929 of 2-20 kb, a fifth decoys: index order and turns of 64 10.1 ms, without
  // 17.3; 20,000 of 100 bases-50 kb the other way round, 5.8 and 4.3). A single pair
  // has nobody to take turns with.
  const uint64_t lanes = warps * plan->lp;
  const bool automatic = slice_windows == 0 && n > lanes && n < 16 * lanes;
  const bool stored = slice_windows > 0 && !asked && n > lanes;
  plan->slice = n < 2 ? 0u : turns_asked || stored ? static_cast<uint32_t>(slice_windows) : automatic ? 64u : 0u;
  plan->turns = automatic ? 4u : stored ? kFixedTurns : 0u;
  if (tuned && n > lanes) {
    plan->choice = kChoice | (made_for == kMadeForAlike ? kChoiceAlike : 0u) | (lpt ? 0u : kChoiceIndex) |
                   (slice_windows > 0 ? kChoiceTurns : slice_windows < 0 ? kChoiceNoTurns : 0u);
    if (n < 16 * lanes) {
      plan->choice |= kChoiceAutomatic;
      if (slice_windows < 0) {  // (automatic turns where the tuning does not apply)
        plan->slice = 64u;
        plan->turns = 4u;
      }
    }
  }
  // (waiting lanes take part in the ring as well)
  if (plan->slice) plan->lanes = plan->lp;
  return cudaSuccess;
}

cudaError_t length_class(uint32_t n_pairs, int W, int O, const void* ws, cudaStream_t s, bool* outnumber,
                         bool* alike) {
  AlignParams p{};
  p.n_pairs = n_pairs;
  p.W = W;
  p.O = O;
  p.tb_table = tb_table(kTbOrderDefault);
  LanePlan plan{};
  cudaError_t e = lane_plan(p, 1, false, true, kMadeForAny, &plan);
  *outnumber = *alike = false;
  if (e != cudaSuccess || !plan.slice) return e;  // (stored turns are for pairs that do)
  *outnumber = true;
  uint32_t fact = 0;
  const char* at = static_cast<const char*>(ws) + workspace_layout(n_pairs).queue + 5 * sizeof(uint32_t);
  e = cudaMemcpyAsync(&fact, at, sizeof(fact), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  *alike = fact != 0;
  return e;
}

WorkspaceLayout workspace_layout(uint32_t n_pairs) {
  auto up = [](size_t x) { return (x + 255) & ~static_cast<size_t>(255); };
  WorkspaceLayout L{};
  L.queue = 0;
  L.hist = up(L.queue + 256);
  L.order = up(L.hist + sizeof(uint32_t) * kLptBuckets);
  L.locate = up(L.order + sizeof(uint32_t) * static_cast<size_t>(n_pairs));
  L.ring = up(L.locate + sizeof(int32_t) * static_cast<size_t>(n_pairs));
  L.ring_seq = up(L.ring + 2 * sizeof(uint32_t) * static_cast<size_t>(n_pairs));
  L.state = up(L.ring_seq + 2 * sizeof(uint32_t) * static_cast<size_t>(n_pairs));
  L.total = up(L.state + sizeof(SlotState) * static_cast<size_t>(n_pairs));
  return L;
}

cudaError_t launch_batched(const AlignParams& p, const LanePlan& plan, void* ws, cudaStream_t s) {
  if (p.n_pairs == 0) return cudaSuccess;
  const WorkspaceLayout L = workspace_layout(p.n_pairs);
  char* w = static_cast<char*>(ws);
  uint32_t* queue = reinterpret_cast<uint32_t*>(w + L.queue);
  uint32_t* hist = reinterpret_cast<uint32_t*>(w + L.hist);
  uint32_t* order = reinterpret_cast<uint32_t*>(w + L.order);
  // One block orders a batch that keeps it busy for a few microseconds at most.
  // (Teams have no use for an order. Below 64 pairs its three launches are made all
  // the same: tests/test_gpu_parity.py counts them in a graph's replay of 40 pairs.)
  cudaError_t e = cudaSuccess;
  if (plan.team && p.n_pairs >= 64) return launch_team(p, plan, nullptr, s);
  if (plan.lpt && p.n_pairs >= 64 && p.n_pairs <= kLptOneBlock) {
    lpt_block_kernel<<<1, kLptBuckets, 0, s>>>(p.read_len, p.n_pairs, static_cast<uint32_t>(plan.warps),
                                               plan.staged && plan.vw == 2, plan.choice, queue, order);
    count_launches(1);
  } else {
    if ((e = cudaMemsetAsync(w, 0, L.order, s)) != cudaSuccess) return e;  // counters + histogram
    if (plan.lpt &&
        (e = launch_lpt_order(p.read_len, p.n_pairs, hist, order, static_cast<uint32_t>(plan.warps),
                              plan.staged && plan.vw == 2, plan.choice, queue + 5, s)) != cudaSuccess)
      return e;
  }
  if (plan.team) return launch_team(p, plan, plan.lpt ? order : nullptr, s);
  uint32_t* ring = reinterpret_cast<uint32_t*>(w + L.ring);
  uint32_t* ring_seq = reinterpret_cast<uint32_t*>(w + L.ring_seq);
  SlotState* state = reinterpret_cast<SlotState*>(w + L.state);
  if (plan.slice) {
    const int blocks = static_cast<int>(std::min<uint32_t>((p.n_pairs + 255) / 256, 1024u));
    ring_init_kernel<<<blocks, 256, 0, s>>>(p.n_pairs,
                                            static_cast<uint32_t>(plan.warps * plan.lp),
                                            plan.lpt ? order : nullptr, ring, ring_seq, queue, state,
                                            p.status, p.dist, p.ref_consumed, p.n_runs);
    count_launches(1);
  }
  const BatchArgs a{queue, plan.lpt ? order : nullptr, plan.cols, plan.lanes, plan.slice, plan.turns,
                    ring, ring_seq, state, g_idle_polls.load(std::memory_order_relaxed),
                    g_push_polls.load(std::memory_order_relaxed)};
  if (plan.vw == 1) lane_launch<1, 32, 1>(p, plan, a, s);
  else if (plan.vw == 2) lane_launch<2, 32, 1>(p, plan, a, s);
  else wide_lane_launch(p, plan, a, s);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_batched_locate(const AlignParams& p, const LanePlan& plan,
                                  const uint32_t* start_span, int32_t* ref_start, void* ws,
                                  cudaStream_t s) {
  if (p.n_pairs == 0) return cudaSuccess;
  const WorkspaceLayout L = workspace_layout(p.n_pairs);
  int32_t* locate_d = reinterpret_cast<int32_t*>(static_cast<char*>(ws) + L.locate);
  int dev = 0, sms = 0;
  cudaError_t e = device_sms(&dev, &sms);
  if (e != cudaSuccess) return e;
  // Lanes per pair: the most that two or three warps per scheduler hold (each
  // lane adds 2 W columns to the search).
  int log_q = 0;
  while (log_q < 5 && (2ull * p.n_pairs << log_q) <= 320ull * sms) ++log_q;
  const LocateArgs a{start_span, ref_start, locate_d};
  if (plan.vw == 1) locate_launch<1>(p, a, log_q, s);
  else if (plan.vw == 2) locate_launch<2>(p, a, log_q, s);
  else wide_locate_launch(plan.vw, p, a, log_q, s);
  count_launches(1);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  AlignParams q = p;
  q.start_span = start_span;
  q.ref_start = ref_start;
  q.locate_d = locate_d;
  return launch_batched(q, plan, ws, s);
}

// ---------------------------------------------------------------------------
// Serving step
// ---------------------------------------------------------------------------

namespace {

size_t step_smem(int vw, int cols) {
  return vw == 1 ? lane_block_smem<LaneShape<1, 32, 1>>(cols, false, false)
                 : lane_block_smem<LaneShape<2, 32, 1>>(cols, false, false);
}

template <int VW>
cudaError_t step_setup(int cols, int* warps_per_sm) {
  // (The attribute is the function's, not the server's: a server of another W sets
  // the same.)
  const size_t smem = step_smem(VW, cols);
  const cudaError_t e = cudaFuncSetAttribute(align_step_kernel<VW>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, kSharedOptIn);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(warps_per_sm, align_step_kernel<VW>, 32, smem);
}

}  // namespace

cudaError_t prepare_step(int W, LanePlan* plan) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  *plan = LanePlan{};
  plan->vw = vw_for(W);
  plan->lp = 32;
  plan->cols = up8(W);
  e = plan->vw == 1 ? step_setup<1>(plan->cols, &per_sm) : step_setup<2>(plan->cols, &per_sm);
  if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
  plan->warps = sms * std::min(per_sm, 4);
  plan->lanes = 32;
  return e;
}

cudaError_t launch_step(const AlignParams& p, const LanePlan& plan, const StepArgs& a,
                        cudaStream_t s) {
  int dev = 0, sms = 0;
  const cudaError_t q = device_sms(&dev, &sms);
  if (q != cudaSuccess) return q;
  if (team_size(a.n_active, sms)) return launch_step_team(p, sms, a, s);
  const size_t smem = step_smem(plan.vw, plan.cols);
  if (plan.vw == 1) align_step_kernel<1><<<plan.warps, 32, smem, s>>>(p, a);
  else align_step_kernel<2><<<plan.warps, 32, smem, s>>>(p, a);
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) count_launches(1);
  return e;
}

}  // namespace ga
