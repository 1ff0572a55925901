// The kernels with many instances, each family compiled into a module of its own (netmax_fused.cu, netmax_tiles_*.cu, netmax_pipe.cu).
// A module is loaded when one of its kernels is first asked for, which takes 2 to 3 ms per megabyte: a process pays for the
// families that its problems run on.  ms for a process's first context and rounds, all instances in one module / so: one round of 4 x 4,096
// elements 68 / 34, 20 rounds of 8 x 600,000 68 / 11, of 64 x 100,000 67 / 31.
#pragma once
#include "netmax_kernels.cuh"
#include "netmax_pipe.cuh"
#include "netmax_tiles.cuh"

namespace netmax {

using FusedKernel = void (*)(const FusedParams);
using TileKernel = void (*)(const TileParams);
using PipeKernel = void (*)(const PipeParams);

// halves: 1 for fp32 state, 2 for bfloat16 state (Philox blocks per 16-byte column group).
// The instance for M workers and launches of `rounds` rounds (all of one M share one layout of the shared memory).
FusedKernel pick_fused_kernel(int objective, int halves, int32_t M, int rounds);
template <bool kBf16>
TileKernel pick_tile_kernel_of(int objective, int rows, int G, int warps);
extern template TileKernel pick_tile_kernel_of<false>(int objective, int rows, int G, int warps);
extern template TileKernel pick_tile_kernel_of<true>(int objective, int rows, int G, int warps);
inline TileKernel pick_tile_kernel(int objective, int halves, int rows, int G, int warps) {
  return halves == 2 ? pick_tile_kernel_of<true>(objective, rows, G, warps) : pick_tile_kernel_of<false>(objective, rows, G, warps);
}
PipeKernel pick_pipe_kernel(int objective, int halves, int rows);

}  // namespace netmax
