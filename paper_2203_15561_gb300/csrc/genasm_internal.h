// Internal launch interface between the C ABI (genasm_capi.cu) and the
// kernels (genasm_align.cu, genasm_aux.cu). Not part of the public ABI.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace ga {

// Records `e` as the calling host thread's last CUDA error (what
// ga_last_cuda_error reports) and maps it to GA_OK or GA_ECUDA.
int cuda_fail(cudaError_t e);
int last_cuda_error();

struct AlignParams {
  const uint8_t* reads;
  const uint64_t* read_off;
  const uint32_t* read_len;
  const uint8_t* refs;
  const uint64_t* ref_off;
  const uint32_t* ref_len;
  uint32_t n_pairs;
  int W, O, kmax;  // kmax = min(k, W): no window needs rows above W
  uint64_t tb_table;  // traceback decision table (tb_table(order) in genasm_window.cuh)
  int32_t* dist;
  int32_t* status;
  int32_t* ref_consumed;
  uint32_t* cigar;
  const uint64_t* cigar_off;
  uint32_t* n_runs;
  uint32_t* n_windows;  // optional
  uint64_t* cells;      // optional
  const uint32_t* cigar_cap;  // optional per-pair CIGAR capacity (else cigar_off[p+1] - cigar_off[p])
  // Free-start first window (set by the locate launcher, else null): the
  // locate kernel writes ref_start (alignment start, -1 when the search found
  // no start within k edits) and locate_d (the search's edit count, -1
  // without a search); the alignment starts at ref_start and counts the
  // search's L * (locate_d + 1) DP entries, L = min(ref_len, start_span + W).
  const uint32_t* start_span;
  int32_t* ref_start;
  int32_t* locate_d;
};

// Launch shape of the batched kernel (one lane per pair, one-warp blocks).
struct LanePlan {
  int vw;          // 32-bit words per window vector
  int lp;          // pairs a warp holds
  int cols;        // columns of a lane's table
  int warps;       // persistent grid size
  int lanes;       // of them, those that take pairs in this launch
  bool any_order;  // a traceback order other than the default
  bool staged;     // the next window's bases copied ahead (see genasm_lane.cuh)
  bool lpt;        // longest-first hand-out
  uint32_t slice;  // windows per turn of the sliced queue (0: off)
  uint32_t turns;  // if not 0: turns only for pairs of about one length, each this
                   // fraction of its pair and `slice` windows at least
  int team;        // lanes of a team (8..32, or 128: a block of four warps); 0: no teams
  uint32_t choice;  // what the ordering decides by the lengths (kChoice*; 0: as ever)
};

// `turns` for turns of `slice` windows whatever the pair's length.
constexpr uint32_t kFixedTurns = 1u << 20;

// A tuning that the autotuner stored, taken on the device where the pairs' lengths
// are of the kind it was made for: of about one length, or mixed.
constexpr uint32_t kChoice = 1, kChoiceAlike = 2;            // made for pairs of about one length
constexpr uint32_t kChoiceIndex = 4;                         // then: index order
constexpr uint32_t kChoiceTurns = 8, kChoiceNoTurns = 16;    // then: turns, none (neither: if automatic)
constexpr uint32_t kChoiceAutomatic = 32;                    // turns pay, of pairs of about one length

// What the lanes of a team take on (see genasm_team.cuh).
constexpr int kTeamLanes = 128;
enum { kTeamLong = 0, kTeamFew = 1, kTeamStrange = 2, kTeamKinds = 3 };
struct TeamStarts {
  uint16_t start[kTeamKinds][kTeamLanes];
};

// Workspace layout of the batched kernel (byte offsets).
struct WorkspaceLayout {
  size_t queue;   // uint32 counters (256 B)
  size_t hist;    // uint32[kLptBuckets]
  size_t order;   // uint32[n_pairs]
  size_t locate;  // int32[n_pairs]: the locate step's edit counts
  size_t ring;    // uint32[2 n_pairs]: slots of the sliced queue's ring
  size_t ring_seq;  // uint32[2 n_pairs]: their sequence numbers
  size_t state;   // SlotState[n_pairs]: window state of pairs between turns
  size_t total;
};

constexpr int kLptBuckets = 1024;

// Saved window state of one pair between serving steps (all zero = fresh).
struct SlotState {
  uint32_t pos_p, pos_t, edits, windows;
  uint64_t cells;
  uint32_t runs, run_op, run_len, pad;
};

struct StepArgs {
  const uint32_t* active;  // slots to advance this step (mapped host memory)
  uint32_t n_active;
  uint32_t windows;        // windows per pair and step
  uint32_t* counters;      // three, zero before a step and after it: work counter,
                           // finished slots, finished warps
  SlotState* state;        // per slot
  uint32_t* done;          // slots that finished this step (mapped host memory)
  uint32_t* n_done;        // their count (mapped host memory)
  int cols;                // columns of a lane's table
};

// prepare_step fills the launch shape of the serving step for windows of W <= 64
// bases and sets the kernel's shared-memory attribute; launch_step launches it.
cudaError_t prepare_step(int W, LanePlan* plan);
// Pairs by teams of lanes (genasm_team.cu): the team for n pairs (0: none), the
// batched launch of plan.team, and the serving step's.
int team_size(uint64_t n, int sms);
cudaError_t launch_step_team(const AlignParams& p, int sms, const StepArgs& a, cudaStream_t s);
cudaError_t launch_team(const AlignParams& p, const LanePlan& plan, const uint32_t* order, cudaStream_t s);
cudaError_t launch_step(const AlignParams& p, const LanePlan& plan, const StepArgs& a,
                        cudaStream_t s);

WorkspaceLayout workspace_layout(uint32_t n_pairs);

// Ablation kernels (genasm_ablation.cu): variant 0..3, see ga_align_ablation.
// Bounds of the sliced queue's waits (polls; 0 = the default of seconds).
void set_queue_wait_limits(uint32_t idle_polls, uint32_t push_polls);
cudaError_t ablation_workspace_bytes(uint32_t n_pairs, int variant, size_t* bytes);
cudaError_t launch_ablation(const AlignParams& p, int variant, uint64_t* table_bytes, void* ws,
                            size_t ws_bytes, cudaStream_t s);

// Longest-read-first order of n pairs (counting sort over kLptBuckets read
// length buckets): hist must hold kLptBuckets zeroed counters, order n entries.
// facts (may be null) receives 1 when the pairs are of about one length, else 0,
// the lanes of each of `warps` warps that they can use, and with `split` how the
// longest are split over the warps (n up to 2^22); `choice` as in LanePlan.
cudaError_t launch_lpt_order(const uint32_t* read_len, uint32_t n, uint32_t* hist, uint32_t* order,
                             uint32_t warps, bool split, uint32_t choice, uint32_t* facts, cudaStream_t s);

// Lanes per warp of the long pairs that decide how long a batch takes (see
// length_split): how many, and their numbers.
constexpr int kSplits = 9;
__host__ __device__ constexpr uint32_t kSplitLanes(int k) {
  constexpr uint32_t lanes[kSplits] = {1, 2, 3, 4, 6, 8, 12, 16, 24};
  return lanes[k];
}

// Kernel launches issued by the library (process-wide counter).
uint64_t launch_count();
void count_launches(uint64_t n);
void uncount_launches(uint64_t n);  // kernels that were captured into a graph, not run

// Per-device tuning chosen by the autotuner (or set by the caller), kept
// apart for the two forms of the batched alignment: mode 0 anchored first
// windows (ga_align_batch), mode 1 free-start first windows
// (ga_align_batch_locate).
// `made_for`: the pairs' lengths that the autotuner had (kMade*).
enum { kMadeForAny = -1, kMadeForMixed = 0, kMadeForAlike = 1 };
bool stored_tuning(int W, int O, int k, struct ga_tuning_s* out, int* made_for, int mode);
void store_tuning(int W, int O, int k, const struct ga_tuning_s* t, int made_for, int mode);

cudaError_t measure_int_peak(double out[3], cudaStream_t s);
cudaError_t measure_smem_peak(double out[2], cudaStream_t s);

size_t compact_workspace_bytes(uint32_t n_pairs);
cudaError_t launch_compact(const uint32_t* cigar, const uint64_t* cigar_off, const uint32_t* n_runs,
                           uint32_t n, uint32_t* out, uint64_t out_cap, uint64_t* out_off, void* ws,
                           cudaStream_t s);

cudaError_t launch_pack(const uint8_t* ascii, uint64_t n, uint8_t* packed, uint32_t* n_invalid,
                        cudaStream_t s);
cudaError_t launch_plain(const AlignParams& p, cudaStream_t s);
cudaError_t launch_batched(const AlignParams& p, const LanePlan& plan, void* ws, cudaStream_t s);

// The batched alignment with a free-start first window: the locate kernel
// over every pair (start spans d_start_span, starts into d_ref_start), then
// the batched kernel starting each pair there.
cudaError_t launch_batched_locate(const AlignParams& p, const LanePlan& plan,
                                  const uint32_t* start_span, int32_t* ref_start, void* ws,
                                  cudaStream_t s);

// The tuning in force for (W, O, k) on the current device: `t` (nullptr: none)
// over the stored one of `mode` over the library's, and what it was made for.
// cudaErrorInvalidValue for one that names no launch shape.
cudaError_t resolve_tuning(int W, int O, int k, const struct ga_tuning_s* t, int mode,
                           struct ga_tuning_s* out, int* made_for);

// Launch shape of the batched kernel for p (p.n_pairs, W, O, order) on the
// current device; slice_windows and lpt as in ga_tuning. `asked`: they come with
// the call, not from a stored tuning; made_for: what that was made for.
cudaError_t lane_plan(const AlignParams& p, int slice_windows, bool asked, bool lpt, int made_for,
                      LanePlan* plan);

// Whether n_pairs outnumber the resident lanes, and whether they are of about one
// length, as an untuned alignment has just left it in the workspace (waits for the
// stream).
cudaError_t length_class(uint32_t n_pairs, int W, int O, const void* ws, cudaStream_t s, bool* outnumber,
                         bool* alike);

}  // namespace ga
