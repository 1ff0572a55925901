// Instances of fused_rounds_kernel.
#include "netmax_instances.h"

namespace netmax {

template <int kReg, bool kStart>
static FusedKernel pick_fused_kernel_r(int objective, int halves) {
  if (halves == 2) return objective == 1 ? fused_rounds_kernel<1, true, kReg, kStart> : fused_rounds_kernel<0, true, kReg, kStart>;
  return objective == 1 ? fused_rounds_kernel<1, false, kReg, kStart> : fused_rounds_kernel<0, false, kReg, kStart>;
}
FusedKernel pick_fused_kernel(int objective, int halves, int32_t M, int rounds) {
  const bool start = M <= kStartWorkers;
  if (rounds <= 4) return start ? pick_fused_kernel_r<4, true>(objective, halves) : pick_fused_kernel_r<4, false>(objective, halves);
  if (rounds <= 8) return start ? pick_fused_kernel_r<8, true>(objective, halves) : pick_fused_kernel_r<8, false>(objective, halves);
  return start ? pick_fused_kernel_r<0, true>(objective, halves) : pick_fused_kernel_r<0, false>(objective, halves);
}

}  // namespace netmax
