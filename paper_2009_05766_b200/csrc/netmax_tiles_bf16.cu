#include "netmax_tile_instances.inc"

template netmax::TileKernel netmax::pick_tile_kernel_of<true>(int objective, int rows, int G, int warps);
