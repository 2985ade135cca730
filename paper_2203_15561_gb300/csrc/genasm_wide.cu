// The batched alignment and the locate step for windows of 65..128 bases:
// genasm_batch.cuh with vectors of three words (up to 96 bases) and four.
#include "genasm_batch.cuh"

namespace ga {

cudaError_t wide_lane_setup(int vw, int cols, bool any_order, int* warps_per_sm) {
  return vw == 3 ? lane_setup_order<3>(cols, any_order, warps_per_sm)
                 : lane_setup_order<4>(cols, any_order, warps_per_sm);
}

void wide_lane_launch(int vw, const AlignParams& p, const LanePlan& plan, const BatchArgs& a,
                      cudaStream_t s) {
  if (vw == 3) lane_launch<3>(p, plan, a, s);
  else lane_launch<4>(p, plan, a, s);
}

void wide_locate_launch(int vw, const AlignParams& p, const LocateArgs& a, int log_q,
                        cudaStream_t s) {
  if (vw == 3) locate_launch<3>(p, a, log_q, s);
  else locate_launch<4>(p, a, log_q, s);
}

}  // namespace ga
