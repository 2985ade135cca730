// C ABI of the library: argument checks, tuning resolution and launches.
// Every entry point validates its arguments before enqueuing anything and
// maps CUDA failures to GA_ECUDA (the CUDA code is kept per host thread).
#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

#include "genasm.h"
#include "genasm_internal.h"
#include "genasm_window.cuh"

namespace ga {

namespace {
thread_local int g_last_cuda = 0;
}  // namespace

int cuda_fail(cudaError_t e) {
  g_last_cuda = static_cast<int>(e);
  return e == cudaSuccess ? GA_OK : GA_ECUDA;
}

int last_cuda_error() { return g_last_cuda; }

}  // namespace ga

namespace {

using ga::cuda_fail;

bool bad_wok(int W, int O, int k) { return W < 1 || W > GA_MAX_W || O < 0 || O >= W || k < 0; }
bool wide_window(int W) { return W > GA_MAX_W_ONCHIP; }

int fill_params(const uint8_t* d_reads, const uint64_t* d_read_off, const uint32_t* d_read_len,
                const uint8_t* d_refs, const uint64_t* d_ref_off, const uint32_t* d_ref_len,
                uint32_t n_pairs, int W, int O, int k, int32_t* d_dist, int32_t* d_status,
                int32_t* d_ref_consumed, uint32_t* d_cigar, const uint64_t* d_cigar_off,
                uint32_t* d_n_runs, uint32_t* d_n_windows, uint64_t* d_cells, ga::AlignParams* p) {
  if (bad_wok(W, O, k)) return GA_EINVAL;
  if (n_pairs > 0 && (!d_reads || !d_read_off || !d_read_len || !d_refs || !d_ref_off ||
                      !d_ref_len || !d_dist || !d_status || !d_ref_consumed || !d_cigar ||
                      !d_cigar_off || !d_n_runs))
    return GA_EINVAL;
  p->reads = d_reads;
  p->read_off = d_read_off;
  p->read_len = d_read_len;
  p->refs = d_refs;
  p->ref_off = d_ref_off;
  p->ref_len = d_ref_len;
  p->n_pairs = n_pairs;
  p->W = W;
  p->O = O;
  p->kmax = k < W ? k : W;
  p->tb_table = ga::tb_table(ga::kTbOrderDefault);
  p->dist = d_dist;
  p->status = d_status;
  p->ref_consumed = d_ref_consumed;
  p->cigar = d_cigar;
  p->cigar_off = d_cigar_off;
  p->n_runs = d_n_runs;
  p->n_windows = d_n_windows;
  p->cells = d_cells;
  return GA_OK;
}

// Windows wider than 64 bases take no tuning.
int resolve(int W, int O, int k, const ga_tuning* t, ga_tuning* out, int* made_for, int mode) {
  if (wide_window(W)) {
    *out = ga_tuning{8, 8, 39, 1, 0, 0};
    *made_for = ga::kMadeForAny;
    return GA_OK;
  }
  const cudaError_t e = ga::resolve_tuning(W, O, k, t, mode, out, made_for);
  return e == cudaErrorInvalidValue ? GA_EINVAL : cuda_fail(e);
}

int workspace_bytes(uint32_t n_pairs, int W, int O, int k, const ga_tuning* t, int mode,
                    size_t* bytes_out) {
  if (!bytes_out || bad_wok(W, O, k)) return GA_EINVAL;
  ga_tuning r;
  int made_for = 0;
  const int rc = resolve(W, O, k, t, &r, &made_for, mode);
  if (rc == GA_OK) *bytes_out = ga::workspace_layout(n_pairs).total;
  return rc;
}

// The checks and the launch shape of a batched call whose parameters are filled.
int plan_batched(const ga::AlignParams& p, int k, const ga_tuning* t, int mode, const void* d_workspace,
                 size_t ws_bytes, ga::LanePlan* plan) {
  ga_tuning r;
  int made_for = 0;
  const int rc = resolve(p.W, p.O, k, t, &r, &made_for, mode);
  if (rc != GA_OK) return rc;
  if (!d_workspace || ws_bytes < ga::workspace_layout(p.n_pairs).total) return GA_ENOSPC;
  return cuda_fail(ga::lane_plan(p, r.slice_windows, t != nullptr, r.lpt > 0, made_for, plan));
}

}  // namespace

extern "C" {

int ga_version(void) { return 100; }

const char* ga_strerror(int code) {
  switch (code) {
    case GA_OK: return "ok";
    case GA_EINVAL: return "invalid argument";
    case GA_ENOSPC: return "workspace or capacity too small";
    case GA_ECUDA: return "CUDA error";
    case GA_ETIMEDOUT: return "bounded wait timed out";
    case GA_ENOMEM: return "memory budget exceeded";
    case GA_EAGAIN: return "nothing ready, or the server's waiting requests are at their limit (step, then retry)";
    default: return "unknown error";
  }
}

int ga_last_cuda_error(void) { return ga::last_cuda_error(); }

int ga_pack_2bit(const uint8_t* d_ascii, uint64_t n_chars, uint8_t* d_packed,
                 uint32_t* d_n_invalid, ga_stream_t stream) {
  if (n_chars > 0 && (!d_ascii || !d_packed)) return GA_EINVAL;
  return cuda_fail(ga::launch_pack(d_ascii, n_chars, d_packed, d_n_invalid,
                                   reinterpret_cast<cudaStream_t>(stream)));
}

int ga_workspace_size(uint32_t n_pairs, int W, int O, int k, size_t* bytes_out) {
  return workspace_bytes(n_pairs, W, O, k, nullptr, 0, bytes_out);
}

int ga_workspace_size_tuned(uint32_t n_pairs, int W, int O, int k, const ga_tuning* tuning,
                            size_t* bytes_out) {
  return workspace_bytes(n_pairs, W, O, k, tuning, 0, bytes_out);
}

uint64_t ga_launch_count(void) { return ga::launch_count(); }

int ga_set_queue_wait_limits(uint32_t idle_polls, uint32_t push_polls) {
  ga::set_queue_wait_limits(idle_polls, push_polls);
  return GA_OK;
}

int ga_cigar_compact_workspace_size(uint32_t n_pairs, size_t* bytes_out) {
  if (!bytes_out) return GA_EINVAL;
  *bytes_out = ga::compact_workspace_bytes(n_pairs);
  return GA_OK;
}

int ga_cigar_compact(const uint32_t* d_cigar, const uint64_t* d_cigar_off, const uint32_t* d_n_runs,
                     uint32_t n_pairs, uint32_t* d_out, uint64_t out_cap, uint64_t* d_out_off,
                     void* d_workspace, size_t ws_bytes, ga_stream_t stream) {
  if (!d_out_off || (n_pairs > 0 && (!d_cigar || !d_cigar_off || !d_n_runs || !d_out)))
    return GA_EINVAL;
  if (!d_workspace || ws_bytes < ga::compact_workspace_bytes(n_pairs)) return GA_ENOSPC;
  return cuda_fail(ga::launch_compact(d_cigar, d_cigar_off, d_n_runs, n_pairs, d_out, out_cap,
                                      d_out_off, d_workspace, reinterpret_cast<cudaStream_t>(stream)));
}

int ga_measure_int_peak(double out[3], ga_stream_t stream) {
  if (!out) return GA_EINVAL;
  return cuda_fail(ga::measure_int_peak(out, reinterpret_cast<cudaStream_t>(stream)));
}

int ga_measure_smem_peak(double out[2], ga_stream_t stream) {
  if (!out) return GA_EINVAL;
  return cuda_fail(ga::measure_smem_peak(out, reinterpret_cast<cudaStream_t>(stream)));
}

int ga_align_batch_tuned(const uint8_t* d_reads, const uint64_t* d_read_off,
                         const uint32_t* d_read_len, const uint8_t* d_refs,
                         const uint64_t* d_ref_off, const uint32_t* d_ref_len, uint32_t n_pairs,
                         int W, int O, int k, int32_t* d_dist, int32_t* d_status,
                         int32_t* d_ref_consumed, uint32_t* d_cigar, const uint64_t* d_cigar_off,
                         uint32_t* d_n_runs, uint32_t* d_n_windows, uint64_t* d_cells,
                         void* d_workspace, size_t ws_bytes, const ga_tuning* tuning,
                         ga_stream_t stream) {
  ga::AlignParams p{};
  int rc = fill_params(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len, n_pairs, W,
                       O, k, d_dist, d_status, d_ref_consumed, d_cigar, d_cigar_off, d_n_runs,
                       d_n_windows, d_cells, &p);
  if (rc != GA_OK) return rc;
  if (n_pairs == 0) return GA_OK;
  ga::LanePlan plan{};
  rc = plan_batched(p, k, tuning, 0, d_workspace, ws_bytes, &plan);
  if (rc != GA_OK) return rc;
  return cuda_fail(ga::launch_batched(p, plan, d_workspace, reinterpret_cast<cudaStream_t>(stream)));
}

int ga_align_batch_order(const uint8_t* d_reads, const uint64_t* d_read_off,
                         const uint32_t* d_read_len, const uint8_t* d_refs,
                         const uint64_t* d_ref_off, const uint32_t* d_ref_len, uint32_t n_pairs,
                         int W, int O, int k, int32_t* d_dist, int32_t* d_status,
                         int32_t* d_ref_consumed, uint32_t* d_cigar, const uint64_t* d_cigar_off,
                         uint32_t* d_n_runs, uint32_t* d_n_windows, uint64_t* d_cells,
                         int tb_order, void* d_workspace, size_t ws_bytes, ga_stream_t stream) {
  // A permutation of the four edge kinds, two bits each.
  unsigned seen = 0;
  for (int q = 0; q < 4; ++q) seen |= 1u << ((static_cast<unsigned>(tb_order) >> (2 * q)) & 3u);
  if (tb_order < 0 || tb_order > 0xFF || seen != 0xFu) return GA_EINVAL;
  ga::AlignParams p{};
  int rc = fill_params(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len, n_pairs, W,
                       O, k, d_dist, d_status, d_ref_consumed, d_cigar, d_cigar_off, d_n_runs,
                       d_n_windows, d_cells, &p);
  if (rc != GA_OK) return rc;
  if (n_pairs == 0) return GA_OK;
  p.tb_table = ga::tb_table(static_cast<uint32_t>(tb_order));
  ga::LanePlan plan{};
  rc = plan_batched(p, k, nullptr, 0, d_workspace, ws_bytes, &plan);
  if (rc != GA_OK) return rc;
  return cuda_fail(ga::launch_batched(p, plan, d_workspace, reinterpret_cast<cudaStream_t>(stream)));
}

int ga_workspace_size_locate(uint32_t n_pairs, int W, int O, int k, const ga_tuning* tuning,
                             size_t* bytes_out) {
  return workspace_bytes(n_pairs, W, O, k, tuning, 1, bytes_out);
}

int ga_align_batch_locate_tuned(const uint8_t* d_reads, const uint64_t* d_read_off,
                                const uint32_t* d_read_len, const uint8_t* d_refs,
                                const uint64_t* d_ref_off, const uint32_t* d_ref_len,
                                uint32_t n_pairs, int W, int O, int k,
                                const uint32_t* d_start_span, int32_t* d_ref_start,
                                int32_t* d_dist, int32_t* d_status, int32_t* d_ref_consumed,
                                uint32_t* d_cigar, const uint64_t* d_cigar_off, uint32_t* d_n_runs,
                                uint32_t* d_n_windows, uint64_t* d_cells, void* d_workspace,
                                size_t ws_bytes, const ga_tuning* tuning, ga_stream_t stream) {
  ga::AlignParams p{};
  int rc = fill_params(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len, n_pairs, W,
                       O, k, d_dist, d_status, d_ref_consumed, d_cigar, d_cigar_off, d_n_runs,
                       d_n_windows, d_cells, &p);
  if (rc != GA_OK) return rc;
  if (n_pairs > 0 && (!d_start_span || !d_ref_start)) return GA_EINVAL;
  if (n_pairs == 0) return GA_OK;
  ga::LanePlan plan{};
  rc = plan_batched(p, k, tuning, 1, d_workspace, ws_bytes, &plan);
  if (rc != GA_OK) return rc;
  return cuda_fail(ga::launch_batched_locate(p, plan, d_start_span, d_ref_start, d_workspace,
                                             reinterpret_cast<cudaStream_t>(stream)));
}

int ga_align_batch_locate(const uint8_t* d_reads, const uint64_t* d_read_off,
                          const uint32_t* d_read_len, const uint8_t* d_refs,
                          const uint64_t* d_ref_off, const uint32_t* d_ref_len, uint32_t n_pairs,
                          int W, int O, int k, const uint32_t* d_start_span, int32_t* d_ref_start,
                          int32_t* d_dist, int32_t* d_status, int32_t* d_ref_consumed,
                          uint32_t* d_cigar, const uint64_t* d_cigar_off, uint32_t* d_n_runs,
                          uint32_t* d_n_windows, uint64_t* d_cells, void* d_workspace,
                          size_t ws_bytes, ga_stream_t stream) {
  return ga_align_batch_locate_tuned(d_reads, d_read_off, d_read_len, d_refs, d_ref_off,
                                     d_ref_len, n_pairs, W, O, k, d_start_span, d_ref_start,
                                     d_dist, d_status, d_ref_consumed, d_cigar, d_cigar_off,
                                     d_n_runs, d_n_windows, d_cells, d_workspace, ws_bytes,
                                     nullptr, stream);
}

int ga_align_batch(const uint8_t* d_reads, const uint64_t* d_read_off, const uint32_t* d_read_len,
                   const uint8_t* d_refs, const uint64_t* d_ref_off, const uint32_t* d_ref_len,
                   uint32_t n_pairs, int W, int O, int k, int32_t* d_dist, int32_t* d_status,
                   int32_t* d_ref_consumed, uint32_t* d_cigar, const uint64_t* d_cigar_off,
                   uint32_t* d_n_runs, uint32_t* d_n_windows, uint64_t* d_cells,
                   void* d_workspace, size_t ws_bytes, ga_stream_t stream) {
  return ga_align_batch_tuned(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len,
                              n_pairs, W, O, k, d_dist, d_status, d_ref_consumed, d_cigar,
                              d_cigar_off, d_n_runs, d_n_windows, d_cells, d_workspace, ws_bytes,
                              nullptr, stream);
}

int ga_ablation_workspace_size(uint32_t n_pairs, int W, int O, int k, int variant,
                               size_t* bytes_out) {
  if (!bytes_out || bad_wok(W, O, k) || wide_window(W) || variant < 0 || variant > 3)
    return GA_EINVAL;
  return cuda_fail(ga::ablation_workspace_bytes(n_pairs, variant, bytes_out));
}

int ga_align_ablation(const uint8_t* d_reads, const uint64_t* d_read_off,
                      const uint32_t* d_read_len, const uint8_t* d_refs, const uint64_t* d_ref_off,
                      const uint32_t* d_ref_len, uint32_t n_pairs, int W, int O, int k,
                      int32_t* d_dist, int32_t* d_status, int32_t* d_ref_consumed,
                      uint32_t* d_cigar, const uint64_t* d_cigar_off, uint32_t* d_n_runs,
                      uint32_t* d_n_windows, uint64_t* d_cells, int variant,
                      uint64_t* d_table_bytes, void* d_workspace, size_t ws_bytes,
                      ga_stream_t stream) {
  if (variant < 0 || variant > 3 || wide_window(W)) return GA_EINVAL;
  ga::AlignParams p{};
  const int rc = fill_params(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len,
                             n_pairs, W, O, k, d_dist, d_status, d_ref_consumed, d_cigar,
                             d_cigar_off, d_n_runs, d_n_windows, d_cells, &p);
  if (rc != GA_OK) return rc;
  if (n_pairs == 0) return GA_OK;
  size_t need = 0;
  const cudaError_t e = ga::ablation_workspace_bytes(n_pairs, variant, &need);
  if (e != cudaSuccess) return cuda_fail(e);
  if (!d_workspace || ws_bytes < need) return GA_ENOSPC;
  return cuda_fail(ga::launch_ablation(p, variant, d_table_bytes, d_workspace, ws_bytes,
                                       reinterpret_cast<cudaStream_t>(stream)));
}

int ga_align_plain(const uint8_t* d_reads, const uint64_t* d_read_off, const uint32_t* d_read_len,
                   const uint8_t* d_refs, const uint64_t* d_ref_off, const uint32_t* d_ref_len,
                   uint32_t n_pairs, int W, int O, int k, int32_t* d_dist, int32_t* d_status,
                   int32_t* d_ref_consumed, uint32_t* d_cigar, const uint64_t* d_cigar_off,
                   uint32_t* d_n_runs, uint32_t* d_n_windows, uint64_t* d_cells,
                   ga_stream_t stream) {
  ga::AlignParams p{};
  const int rc = fill_params(d_reads, d_read_off, d_read_len, d_refs, d_ref_off, d_ref_len,
                             n_pairs, W, O, k, d_dist, d_status, d_ref_consumed, d_cigar,
                             d_cigar_off, d_n_runs, d_n_windows, d_cells, &p);
  if (rc != GA_OK) return rc;
  if (wide_window(W) || n_pairs > 0x7fffffffu) return GA_EINVAL;  // on-chip tables; block per pair
  return cuda_fail(ga::launch_plain(p, reinterpret_cast<cudaStream_t>(stream)));
}

}  // extern "C"
