// Instances of pipe_rounds_kernel.
#include "netmax_instances.h"

namespace netmax {

template <int kRows>
static PipeKernel pick_pipe_kernel_r(int objective, int halves) {
  if (halves == 2) return objective == 1 ? pipe_rounds_kernel<1, true, kRows> : pipe_rounds_kernel<0, true, kRows>;
  return objective == 1 ? pipe_rounds_kernel<1, false, kRows> : pipe_rounds_kernel<0, false, kRows>;
}
PipeKernel pick_pipe_kernel(int objective, int halves, int rows) {
  switch (rows) {
    case 1: return pick_pipe_kernel_r<1>(objective, halves);
    case 2: return pick_pipe_kernel_r<2>(objective, halves);
    case 3: return pick_pipe_kernel_r<3>(objective, halves);
    case 4: return pick_pipe_kernel_r<4>(objective, halves);
    case 5: return pick_pipe_kernel_r<5>(objective, halves);
    case 6: return pick_pipe_kernel_r<6>(objective, halves);
    case 7: return pick_pipe_kernel_r<7>(objective, halves);
    default: return pick_pipe_kernel_r<8>(objective, halves);
  }
}

}  // namespace netmax
