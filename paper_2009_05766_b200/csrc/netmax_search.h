// Index arithmetic of sample_rows_kernel's search: rows of thresholds in shared memory, every sixteenth threshold
// in an implicit search tree beside them.  Plain C++ for a host compiler too.
#pragma once
#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define NM_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define NM_HOST_DEVICE inline
#endif

namespace netmax {

NM_HOST_DEVICE uint32_t sample_levels(uint32_t M) {  // of the tree: 2^levels >= blocks of sixteen
  uint32_t h = 0;
  while ((16u << h) < M) ++h;
  return h;
}
// Words between the rows and between the trees of a CTA: rows start in different banks.
NM_HOST_DEVICE uint32_t sample_stride(uint32_t M, int rows) { return ((M + 31u) & ~31u) + 32u / rows; }
NM_HOST_DEVICE uint32_t sample_tree(uint32_t M, int rows) { return (1u << sample_levels(M)) + 32u / rows; }
NM_HOST_DEVICE size_t sample_smem(uint32_t M, int rows) { return (size_t)rows * (sample_stride(M, rows) + sample_tree(M, rows)) * 4u; }

// Node (from 1 on, children 2n and 2n + 1) of the last threshold before block j, 0 < j < 2^h; z: j's lowest set bit.
NM_HOST_DEVICE uint32_t sample_node(uint32_t j, uint32_t h, uint32_t z) { return (1u << (h - 1 - z)) + (j >> (z + 1)); }
// The block that the search goes on in from leaf 2^h ... 2^(h+1) - 1: never one behind the row's last.
NM_HOST_DEVICE uint32_t sample_block(uint32_t leaf, uint32_t h, uint32_t M) {
  const uint32_t block = leaf - (1u << h), last = (M - 1u) / 16u;
  return block < last ? block : last;
}

}  // namespace netmax
