#include "netmax_tile_instances.inc"

template netmax::TileKernel netmax::pick_tile_kernel_of<false>(int objective, int rows, int G, int warps);
