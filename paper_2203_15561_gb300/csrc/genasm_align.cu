// The batched alignment: pair order, ring set-up, launch shapes and launches
// (the kernels are in genasm_batch.cuh), and the server's step.
#include <algorithm>
#include <atomic>
#include <cstdint>

#include <cuda_runtime.h>

#include "genasm.h"
#include "genasm_batch.cuh"
#include "genasm_internal.h"

namespace ga {

// Default bounds of the two waits (ga_set_queue_wait_limits changes them):
// polls of a warp whose groups all wait for a pair (about 0.2 microseconds
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

__global__ void lpt_histogram_kernel(const uint32_t* __restrict__ read_len, uint32_t n,
                                     uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[kLptBuckets];
  for (int x = threadIdx.x; x < kLptBuckets; x += blockDim.x) h[x] = 0;
  __syncthreads();
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x)
    atomicAdd(&h[lpt_bucket(read_len[q])], 1u);
  __syncthreads();
  for (int x = threadIdx.x; x < kLptBuckets; x += blockDim.x)
    if (h[x]) atomicAdd(&hist[x], h[x]);
}

// Exclusive scan of the bucket counts in place (one block of kLptBuckets threads).
__global__ void lpt_scan_kernel(uint32_t* hist) {
  __shared__ uint32_t s[kLptBuckets];
  const int x = threadIdx.x;
  const uint32_t v = hist[x];
  s[x] = v;
  __syncthreads();
  for (int off = 1; off < kLptBuckets; off <<= 1) {
    const uint32_t add = x >= off ? s[x - off] : 0u;
    __syncthreads();
    s[x] += add;
    __syncthreads();
  }
  hist[x] = s[x] - v;
}

__global__ void lpt_scatter_kernel(const uint32_t* __restrict__ read_len, uint32_t n,
                                   uint32_t* __restrict__ cursor, uint32_t* __restrict__ order) {
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const uint32_t pos = atomicAdd(&cursor[lpt_bucket(read_len[q])], 1u);
    order[pos] = q;
  }
}

cudaError_t launch_lpt_order(const uint32_t* read_len, uint32_t n, uint32_t* hist, uint32_t* order,
                             cudaStream_t s) {
  const int blocks = static_cast<int>(std::min<uint32_t>((n + 255) / 256, 1024u));
  lpt_histogram_kernel<<<blocks, 256, 0, s>>>(read_len, n, hist);
  lpt_scan_kernel<<<1, kLptBuckets, 0, s>>>(hist);
  lpt_scatter_kernel<<<blocks, 256, 0, s>>>(read_len, n, hist, order);
  count_launches(3);
  return cudaGetLastError();
}

// The ring of the sliced queue (2n slots) starts with every pair: slot x < n
// holds hand-out position x (the LPT order, or pair x), published with
// sequence number x + 1; slots n..2n-1 are free for positions n..2n-1. Every
// pair starts as timed out (distance and reference end -1, no runs): a pair
// that finishes overwrites it, and one left in the ring when a bounded wait
// ran out keeps it.
__global__ void ring_init_kernel(uint32_t n, const uint32_t* __restrict__ order,
                                 uint32_t* __restrict__ ring, uint32_t* __restrict__ seq,
                                 uint32_t* __restrict__ queue, int32_t* __restrict__ status,
                                 int32_t* __restrict__ dist, int32_t* __restrict__ ref_consumed,
                                 uint32_t* __restrict__ n_runs) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    queue[2] = n;  // tail: the ring starts with every pair
    queue[3] = n;  // pairs not finished
  }
  for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < 2u * n; x += gridDim.x * blockDim.x) {
    if (x < n) {
      ring[x] = order ? order[x] : x;
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

cudaError_t resolve_tuning(int W, int O, int k, const ga_tuning* t, int mode, ga_tuning* out) {
  ga_tuning d{8, 8, 39, 1, 0, 0};
  stored_tuning(W, O, k, &d, mode);  // chosen by an autotuner or set by ga_tuning_set
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

cudaError_t setup_for(int vw, int cols, bool any_order, int* warps_per_sm) {
  if (vw == 1) return lane_setup_order<1>(cols, any_order, warps_per_sm);
  if (vw == 2) return lane_setup_order<2>(cols, any_order, warps_per_sm);
  return wide_lane_setup(vw, cols, any_order, warps_per_sm);
}

}  // namespace

cudaError_t lane_plan(const AlignParams& p, int slice_windows, bool lpt, LanePlan* plan) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int vw = vw_for(p.W);
  plan->vw = vw;
  plan->any_order = p.tb_table != tb_table(kTbOrderDefault);
  plan->lpt = lpt;
  // A table of every column a last window walks when four warps of them fit an
  // SM, else of the W - O columns of the other windows.
  int per_sm = 0;
  plan->cols = up8(p.W);
  if ((e = setup_for(vw, plan->cols, plan->any_order, &per_sm)) != cudaSuccess) return e;
  if (per_sm < 4) {
    plan->cols = up8(p.W - p.O);
    if ((e = setup_for(vw, plan->cols, plan->any_order, &per_sm)) != cudaSuccess) return e;
  }
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  // One warp per scheduler while its lanes hold every pair, else all that fit.
  const uint64_t n = std::max<uint32_t>(p.n_pairs, 1);
  uint64_t warps = static_cast<uint64_t>(sms) * std::min(per_sm, 4);
  if (n > 32 * warps) warps = static_cast<uint64_t>(sms) * per_sm;
  warps = std::min(warps, n);
  plan->warps = static_cast<int>(warps);
  plan->lanes = static_cast<int>(std::min<uint64_t>(32, (n + warps - 1) / warps));
  // Windows per turn of the sliced queue: the tuning's choice, else turns of 64
  // windows when the pairs outnumber the resident lanes less than 16 times over
  // (more pairs than that leave a tail of under a sixteenth of a round). A
  // single pair has nobody to take turns with.
  const uint64_t lanes = warps * 32;
  plan->slice = slice_windows < 0 || n < 2 ? 0u
                : slice_windows > 0       ? static_cast<uint32_t>(slice_windows)
                : n > lanes && n < 16 * lanes ? 64u
                                              : 0u;
  return cudaSuccess;
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
  cudaError_t e = cudaMemsetAsync(w, 0, L.order, s);  // counters + histogram
  if (e != cudaSuccess) return e;
  if (plan.lpt && (e = launch_lpt_order(p.read_len, p.n_pairs, hist, order, s)) != cudaSuccess)
    return e;
  uint32_t* ring = reinterpret_cast<uint32_t*>(w + L.ring);
  uint32_t* ring_seq = reinterpret_cast<uint32_t*>(w + L.ring_seq);
  SlotState* state = reinterpret_cast<SlotState*>(w + L.state);
  if (plan.slice) {
    if ((e = cudaMemsetAsync(state, 0, sizeof(SlotState) * p.n_pairs, s)) != cudaSuccess) return e;
    const int blocks = static_cast<int>(std::min<uint32_t>((p.n_pairs + 255) / 256, 1024u));
    ring_init_kernel<<<blocks, 256, 0, s>>>(p.n_pairs, plan.lpt ? order : nullptr, ring,
                                            ring_seq, queue, p.status, p.dist,
                                            p.ref_consumed, p.n_runs);
    count_launches(1);
  }
  const BatchArgs a{queue, plan.lpt ? order : nullptr, plan.cols, plan.lanes, plan.slice, ring,
                    ring_seq, state, g_idle_polls.load(std::memory_order_relaxed),
                    g_push_polls.load(std::memory_order_relaxed)};
  if (plan.vw == 1) lane_launch<1>(p, plan, a, s);
  else if (plan.vw == 2) lane_launch<2>(p, plan, a, s);
  else wide_lane_launch(plan.vw, p, plan, a, s);
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
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  // Lanes per pair: as many as one warp per scheduler has for every pair.
  int log_q = 0;
  while (log_q < 5 && (static_cast<uint64_t>(p.n_pairs) << log_q) <= 128ull * sms) ++log_q;
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

template <int VW>
cudaError_t step_setup(int cols, int* warps_per_sm) {
  const size_t smem = lane_block_smem(VW, cols, false);
  cudaError_t e = cudaFuncSetAttribute(align_step_kernel<VW>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
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
  plan->cols = up8(W);
  e = plan->vw == 1 ? step_setup<1>(plan->cols, &per_sm) : step_setup<2>(plan->cols, &per_sm);
  if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
  plan->warps = sms * std::min(per_sm, 4);
  plan->lanes = 32;
  return e;
}

cudaError_t launch_step(const AlignParams& p, const LanePlan& plan, const StepArgs& a,
                        cudaStream_t s) {
  const size_t smem = lane_block_smem(plan.vw, plan.cols, false);
  if (plan.vw == 1) align_step_kernel<1><<<plan.warps, 32, smem, s>>>(p, a);
  else align_step_kernel<2><<<plan.warps, 32, smem, s>>>(p, a);
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) count_launches(1);
  return e;
}

// The finished count and the finished slots of a step, into host-mapped memory
// (one block; the host reads them once the step's event has completed).
__global__ void step_copyout_kernel(const uint32_t* __restrict__ counters,
                                    const uint32_t* __restrict__ done, uint32_t* host_count,
                                    uint32_t* host_done) {
  const uint32_t nd = counters[1];
  for (uint32_t q = threadIdx.x; q < nd; q += blockDim.x) host_done[q] = done[q];
  if (threadIdx.x == 0) host_count[0] = nd;
}

cudaError_t launch_step_copyout(const uint32_t* counters, const uint32_t* done,
                                uint32_t* host_count, uint32_t* host_done, cudaStream_t s) {
  step_copyout_kernel<<<1, 256, 0, s>>>(counters, done, host_count, host_done);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace ga
