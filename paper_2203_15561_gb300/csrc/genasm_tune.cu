// Autotuner and CUDA-graph capture of the batched alignment step.
//
// Autotuner: how fast a batch runs whose pairs outnumber the resident lanes depends
// on the order in which they are handed out and on the windows per turn of the
// sliced queue. ga_autotune times a candidate set on the caller's batch with CUDA
// events and stores the best as the default for (device, W, O, k), with the kind of
// lengths that the batch had; ga_align_batch uses it from then on for batches of
// that kind whose pairs outnumber the lanes.
//
// Graph: ga_graph_create captures one whole step (2-bit packing of the ASCII
// inputs, the workspace reset, the longest-first ordering and the alignment
// kernel) into a CUDA graph for fixed buffers; ga_graph_launch replays it with
// one call.
#include <map>
#include <mutex>
#include <tuple>

#include <cuda_runtime.h>

#include "genasm.h"
#include "genasm_internal.h"
#include "genasm_window.cuh"

namespace ga {

namespace {

struct TuneKey {
  int dev, W, O, k, mode;
  bool operator<(const TuneKey& o) const {
    return std::tie(dev, W, O, k, mode) < std::tie(o.dev, o.W, o.O, o.k, o.mode);
  }
};

struct Stored {
  ga_tuning tuning;
  int made_for;
};

std::mutex g_tune_mutex;
std::map<TuneKey, Stored> g_tuned;
thread_local const Stored* g_trial = nullptr;  // an autotuner's candidate, as if stored

}  // namespace

bool stored_tuning(int W, int O, int k, ga_tuning* out, int* made_for, int mode) {
  if (g_trial) {
    *out = g_trial->tuning;
    *made_for = g_trial->made_for;
    return true;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  auto it = g_tuned.find(TuneKey{dev, W, O, k, mode});
  if (it == g_tuned.end()) return false;
  *out = it->second.tuning;
  *made_for = it->second.made_for;
  return true;
}

void store_tuning(int W, int O, int k, const ga_tuning* t, int made_for, int mode) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  std::lock_guard<std::mutex> lock(g_tune_mutex);
  if (t) g_tuned[TuneKey{dev, W, O, k, mode}] = Stored{*t, made_for};
  else g_tuned.erase(TuneKey{dev, W, O, k, mode});
}

}  // namespace ga

namespace {

int bad_wok(int W, int O, int k) {
  return W < 1 || W > GA_MAX_W_ONCHIP || O < 0 || O >= W || k < 0;
}

// The library's own choice: lpt 1, slice_windows 0.
ga_tuning tuning_of(int lpt, int slice_windows) { return ga_tuning{8, 8, 39, lpt, 0, slice_windows}; }

// What another choice has to gain over the library's own to be stored: single runs
// of one tuning differ by up to 2% (24,000 pairs of 10 kb: 2.52-2.57 ms).
constexpr float kGain = 0.98f;

}  // namespace

extern "C" int ga_tuning_get(int W, int O, int k, ga_tuning* out) {
  if (!out || bad_wok(W, O, k)) return GA_EINVAL;
  int made_for = 0;
  if (ga::stored_tuning(W, O, k, out, &made_for, 0)) return GA_OK;
  *out = tuning_of(1, 0);
  return GA_OK;
}

extern "C" int ga_tuning_set(int W, int O, int k, const ga_tuning* t) {
  if (bad_wok(W, O, k)) return GA_EINVAL;
  if (t) {
    size_t bytes = 0;
    const int rc = ga_workspace_size_tuned(1, W, O, k, t, &bytes);  // validates it
    if (rc != GA_OK) return rc;
  }
  ga::store_tuning(W, O, k, t, ga::kMadeForAny, 0);
  return GA_OK;
}

extern "C" int ga_autotune_workspace_size(uint32_t n_pairs, int W, int O, int k, size_t* bytes) {
  if (!bytes || bad_wok(W, O, k)) return GA_EINVAL;
  // (the size does not depend on the tuning)
  return ga_workspace_size(n_pairs, W, O, k, bytes);
}

namespace {

// One alignment of the batch: the anchored form (start_span == nullptr) or
// the free-start form, with an explicit tuning (nullptr: the stored one).
int align_once(const uint8_t* d_reads, const uint64_t* d_read_off, const uint32_t* d_read_len,
               const uint8_t* d_refs, const uint64_t* d_ref_off, const uint32_t* d_ref_len,
               uint32_t n_pairs, int W, int O, int k, const uint32_t* d_start_span,
               int32_t* d_ref_start, int32_t* d_dist, int32_t* d_status, int32_t* d_ref_consumed,
               uint32_t* d_cigar, const uint64_t* d_cigar_off, uint32_t* d_n_runs,
               uint32_t* d_n_windows, uint64_t* d_cells, void* d_workspace, size_t ws_bytes,
               const ga_tuning* t, ga_stream_t stream) {
  if (d_start_span)
    return ga_align_batch_locate_tuned(d_reads, d_read_off, d_read_len, d_refs, d_ref_off,
                                       d_ref_len, n_pairs, W, O, k, d_start_span, d_ref_start,
                                       d_dist, d_status, d_ref_consumed, d_cigar, d_cigar_off,
                                       d_n_runs, d_n_windows, d_cells, d_workspace, ws_bytes, t,
                                       stream);
  return ga_align_batch_tuned(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len,
                              n_pairs, W, O, k, d_dist, d_status, d_ref_consumed, d_cigar,
                              d_cigar_off, d_n_runs, d_n_windows, d_cells, d_workspace, ws_bytes, t,
                              stream);
}

int autotune(const uint8_t* d_reads, const uint64_t* d_read_off, const uint32_t* d_read_len,
             const uint8_t* d_refs, const uint64_t* d_ref_off, const uint32_t* d_ref_len,
             uint32_t n_pairs, int W, int O, int k, const uint32_t* d_start_span,
             int32_t* d_ref_start, int32_t* d_dist, int32_t* d_status, int32_t* d_ref_consumed,
             uint32_t* d_cigar, const uint64_t* d_cigar_off, uint32_t* d_n_runs,
             uint32_t* d_n_windows, uint64_t* d_cells, void* d_workspace, size_t ws_bytes,
             ga_tuning* best, float* best_ms, ga_stream_t stream) {
  if (bad_wok(W, O, k) || n_pairs == 0 || !d_n_windows || !d_cells) return GA_EINVAL;
  const bool locate = d_start_span != nullptr;
  const int mode = locate ? 1 : 0;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // One run with statistics: they are part of the call's outputs.
  int rc = align_once(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len, n_pairs, W, O,
                      k, d_start_span, d_ref_start, d_dist, d_status, d_ref_consumed, d_cigar,
                      d_cigar_off, d_n_runs, d_n_windows, d_cells, d_workspace, ws_bytes, nullptr,
                      stream);
  if (rc != GA_OK) return rc;

  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) return GA_ECUDA;
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return GA_ECUDA;
  }
  // One warm-up run, then one timed run, as if it were stored already.
  const auto time_of = [&](const ga::Stored& c, float* ms) -> int {
    ga::g_trial = &c;
    int r = GA_OK;
    for (int run = 0; run < 2 && r == GA_OK; ++run) {
      if (run == 1) cudaEventRecord(e0, s);
      r = align_once(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len, n_pairs, W, O, k,
                     d_start_span, d_ref_start, d_dist, d_status, d_ref_consumed, d_cigar, d_cigar_off,
                     d_n_runs, nullptr, nullptr, d_workspace, ws_bytes, nullptr, stream);
    }
    ga::g_trial = nullptr;
    if (r != GA_OK) return r;
    cudaEventRecord(e1, s);
    if (cudaEventSynchronize(e1) != cudaSuccess) return GA_ECUDA;
    return cudaEventElapsedTime(ms, e0, e1) == cudaSuccess ? GA_OK : GA_ECUDA;
  };
  ga::Stored best_c{tuning_of(1, 0), ga::kMadeForAny};
  float best_t = 0;
  rc = time_of(best_c, &best_t);
  bool outnumber = false, alike = false;
  if (rc == GA_OK) rc = ga::cuda_fail(ga::length_class(n_pairs, W, O, d_workspace, s, &outnumber, &alike));
  if (outnumber) {
    const float library = best_t;
    for (const int lpt : {1, -1})
      for (const int slice : {0, -1, 32, 64, 128}) {
        if (lpt == 1 && slice == 0) continue;
        const ga::Stored c{tuning_of(lpt, slice), alike ? ga::kMadeForAlike : ga::kMadeForMixed};
        float ms = 0;
        if (rc == GA_OK) rc = time_of(c, &ms);
        if (rc == GA_OK && ms < best_t && ms < kGain * library) {
          best_t = ms;
          best_c = c;
        }
      }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != GA_OK) return rc;
  ga::store_tuning(W, O, k, &best_c.tuning, best_c.made_for, mode);
  if (best) *best = best_c.tuning;
  if (best_ms) *best_ms = best_t;
  return GA_OK;
}

}  // namespace

extern "C" int ga_autotune(const uint8_t* d_reads, const uint64_t* d_read_off,
                           const uint32_t* d_read_len, const uint8_t* d_refs,
                           const uint64_t* d_ref_off, const uint32_t* d_ref_len, uint32_t n_pairs,
                           int W, int O, int k, int32_t* d_dist, int32_t* d_status,
                           int32_t* d_ref_consumed, uint32_t* d_cigar, const uint64_t* d_cigar_off,
                           uint32_t* d_n_runs, uint32_t* d_n_windows, uint64_t* d_cells,
                           void* d_workspace, size_t ws_bytes, ga_tuning* best, float* best_ms,
                           ga_stream_t stream) {
  return autotune(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len, n_pairs, W, O, k,
                  nullptr, nullptr, d_dist, d_status, d_ref_consumed, d_cigar, d_cigar_off,
                  d_n_runs, d_n_windows, d_cells, d_workspace, ws_bytes, best, best_ms, stream);
}

extern "C" int ga_autotune_locate(const uint8_t* d_reads, const uint64_t* d_read_off,
                                  const uint32_t* d_read_len, const uint8_t* d_refs,
                                  const uint64_t* d_ref_off, const uint32_t* d_ref_len,
                                  uint32_t n_pairs, int W, int O, int k,
                                  const uint32_t* d_start_span, int32_t* d_ref_start,
                                  int32_t* d_dist, int32_t* d_status, int32_t* d_ref_consumed,
                                  uint32_t* d_cigar, const uint64_t* d_cigar_off,
                                  uint32_t* d_n_runs, uint32_t* d_n_windows, uint64_t* d_cells,
                                  void* d_workspace, size_t ws_bytes, ga_tuning* best,
                                  float* best_ms, ga_stream_t stream) {
  if (!d_start_span || !d_ref_start) return GA_EINVAL;
  return autotune(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len, n_pairs, W, O, k,
                  d_start_span, d_ref_start, d_dist, d_status, d_ref_consumed, d_cigar,
                  d_cigar_off, d_n_runs, d_n_windows, d_cells, d_workspace, ws_bytes, best,
                  best_ms, stream);
}

// ---------------------------------------------------------------------------
// CUDA graph of one step
// ---------------------------------------------------------------------------

struct ga_graph {
  cudaGraph_t graph;
  cudaGraphExec_t exec;
  uint64_t kernels;  // kernels one replay launches
};

extern "C" int ga_graph_create(const uint8_t* d_ascii_reads, uint64_t n_read_chars,
                               const uint8_t* d_ascii_refs, uint64_t n_ref_chars,
                               uint8_t* d_reads, const uint64_t* d_read_off,
                               const uint32_t* d_read_len, uint8_t* d_refs,
                               const uint64_t* d_ref_off, const uint32_t* d_ref_len,
                               uint32_t n_pairs, int W, int O, int k, int32_t* d_dist,
                               int32_t* d_status, int32_t* d_ref_consumed, uint32_t* d_cigar,
                               const uint64_t* d_cigar_off, uint32_t* d_n_runs,
                               uint32_t* d_n_windows, uint64_t* d_cells, void* d_workspace,
                               size_t ws_bytes, const ga_tuning* tuning, ga_graph** out) {
  if (!out || bad_wok(W, O, k) || n_pairs == 0) return GA_EINVAL;
  if ((d_ascii_reads == nullptr) != (d_ascii_refs == nullptr)) return GA_EINVAL;
  // Validate and resolve the tuning outside the capture (it sets kernel attributes).
  size_t need = 0;
  int rc = ga_workspace_size_tuned(n_pairs, W, O, k, tuning, &need);
  if (rc != GA_OK) return rc;
  if (!d_workspace || ws_bytes < need) return GA_ENOSPC;
  cudaStream_t s;
  if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) return GA_ECUDA;
  const uint64_t before = ga_launch_count();
  rc = GA_OK;
  if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) rc = GA_ECUDA;
  if (rc == GA_OK && d_ascii_reads) {
    rc = ga_pack_2bit(d_ascii_reads, n_read_chars, d_reads, nullptr, reinterpret_cast<ga_stream_t>(s));
    if (rc == GA_OK)
      rc = ga_pack_2bit(d_ascii_refs, n_ref_chars, d_refs, nullptr, reinterpret_cast<ga_stream_t>(s));
  }
  if (rc == GA_OK)
    rc = ga_align_batch_tuned(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len, n_pairs,
                              W, O, k, d_dist, d_status, d_ref_consumed, d_cigar, d_cigar_off,
                              d_n_runs, d_n_windows, d_cells, d_workspace, ws_bytes, tuning,
                              reinterpret_cast<ga_stream_t>(s));
  cudaGraph_t graph = nullptr;
  const cudaError_t ee = cudaStreamEndCapture(s, &graph);
  cudaStreamDestroy(s);
  if (rc != GA_OK || ee != cudaSuccess || graph == nullptr) {
    if (graph) cudaGraphDestroy(graph);
    cudaGetLastError();
    return rc != GA_OK ? rc : GA_ECUDA;
  }
  cudaGraphExec_t exec = nullptr;
  if (cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) {
    cudaGraphDestroy(graph);
    return GA_ECUDA;
  }
  const uint64_t captured = ga_launch_count() - before;
  ga::uncount_launches(captured);  // captured, not run: counted at each replay instead
  ga_graph* g = new ga_graph{graph, exec, captured};
  *out = g;
  return GA_OK;
}

extern "C" int ga_graph_launch(ga_graph* g, ga_stream_t stream) {
  if (!g) return GA_EINVAL;
  if (cudaGraphLaunch(g->exec, reinterpret_cast<cudaStream_t>(stream)) != cudaSuccess)
    return GA_ECUDA;
  ga::count_launches(g->kernels);
  return GA_OK;
}

extern "C" int ga_graph_destroy(ga_graph* g) {
  if (!g) return GA_OK;
  cudaGraphExecDestroy(g->exec);
  cudaGraphDestroy(g->graph);
  delete g;
  return GA_OK;
}
