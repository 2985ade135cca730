// The batched alignment and the locate step for windows of 65..128 bases:
// genasm_batch.cuh with vectors of three words (up to 96 bases) and four.
#include "genasm_batch.cuh"

namespace ga {

// Pairs per warp: 8 (four lanes each), or 16 or 32 with a lane each.
#define GA_WIDE(plan, call)                                                                      \
  ((plan).vw == 3 ? ((plan).lp == 8 ? call(3, 8, 4) : (plan).lp == 16 ? call(3, 16, 1) : call(3, 32, 1)) \
                  : ((plan).lp == 8 ? call(4, 8, 4) : (plan).lp == 16 ? call(4, 16, 1) : call(4, 32, 1)))

cudaError_t wide_lane_setup(const LanePlan& plan, int* warps_per_sm) {
#define GA_CALL(w, l, n) lane_setup_order<w, l, n>(plan, warps_per_sm)
  return GA_WIDE(plan, GA_CALL);
#undef GA_CALL
}

void wide_lane_launch(const AlignParams& p, const LanePlan& plan, const BatchArgs& a,
                      cudaStream_t s) {
#define GA_CALL(w, l, n) lane_launch<w, l, n>(p, plan, a, s)
  GA_WIDE(plan, GA_CALL);
#undef GA_CALL
}
#undef GA_WIDE

void wide_locate_launch(int vw, const AlignParams& p, const LocateArgs& a, int log_q,
                        cudaStream_t s) {
  if (vw == 3) locate_launch<3>(p, a, log_q, s);
  else locate_launch<4>(p, a, log_q, s);
}

}  // namespace ga
