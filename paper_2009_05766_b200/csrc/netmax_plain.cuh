// Kernels beside the rounds themselves.
//
//   sample_peers_kernel   Algorithm 2, peer selection: one Philox draw per (round, worker)
//                         searched in that worker's row of 32-bit cumulative thresholds
//                         (sample_rows_kernel: many rounds of many workers).
//   sum_*_kernel          telemetry of launches that leave it in parts.
//   init_normal_kernel    x(0) and c from the seed.
//   gather_columns_kernel sampled read-back; narrow_rows_kernel, widen_rows_kernel: bfloat16 state and fp32 hosts.
#pragma once
#include "netmax_kernels.cuh"
#include "netmax_search.h"

namespace netmax {

// ------------------------------------------------------------------------- sampler
struct SampleParams {
  const uint32_t* thresholds;  // [M][M] non-decreasing per row
  const int32_t* last_nz;      // [M] last index with p > 0
  int32_t* out;                // slot s of round r is out + ((slot0 + r) % ring) * M
  int2* draws;                 // same indexing: (peer, bits of the pull weight, 0 on a self-draw); may be NULL
  int32_t* host_out;           // same indexing: mirror in page-locked host memory; may be NULL
  const float* wtab;           // [M][M] pull weights (read when draws is given)
  int64_t slot0, ring;
  uint64_t first_round;
  int64_t n_rounds;
  int32_t M;
  PhiloxKeys keys;
};

__device__ __forceinline__ uint32_t peer_word(const SampleParams& p, uint32_t worker, uint64_t round) {
  return philox4x32_10(0u, worker, (uint32_t)round, philox_ctr3(kTagPeer, round), p.keys).x;
}
__device__ __forceinline__ void put_draw(const SampleParams& p, uint32_t r, uint32_t i, int32_t m) {
  int64_t slot = p.slot0 + r;  // (a batch is never longer than the ring)
  if (slot >= p.ring) slot -= p.ring;
  const int64_t at = slot * p.M + i;
  p.out[at] = m;
  if (p.host_out) p.host_out[at] = m;
  if (p.draws) p.draws[at] = make_int2(m, __float_as_int((m == (int32_t)i) ? 0.0f : __ldg(p.wtab + (size_t)i * p.M + m)));
}

// m = min(#{j : T[j] <= u}, last_nz): the count is found by bisection (T is sorted).  One thread per draw,
// thresholds through the caches: for few rounds or few workers.  At most 2^31 draws per launch.
__global__ void __launch_bounds__(256) sample_peers_kernel(const SampleParams p) {
  launch_dependents();
  const uint32_t M = (uint32_t)p.M, total = (uint32_t)p.n_rounds * M;
  for (uint32_t idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    const uint32_t r = idx / M, i = idx - r * M;
    const uint32_t u = peer_word(p, i, p.first_round + r);
    const uint32_t* __restrict__ row = p.thresholds + (size_t)i * M;
    int32_t lo = 0, hi = p.M;
    while (lo < hi) {
      const int32_t mid = (lo + hi) >> 1;
      if (__ldg(row + mid) <= u) lo = mid + 1; else hi = mid;
    }
    put_draw(p, r, i, min(lo, __ldg(p.last_nz + i)));
  }
}

// The same for many rounds of many workers: bisection through the caches is twelve dependent trips to L2 per draw
// (177 us for 1,024 rounds of 4,096 workers).  Here a CTA brings the rows of kSampleRows workers into shared
// memory, once and in whole lines, and draws for them in all rounds of its share.  Lanes run over workers first, so
// that a round's draws leave as segments.  In sorted order the probes of a bisection are a power of two apart, all in
// one bank (42 us of conflicts and waiting); so every sixteenth threshold is copied into an implicit search tree, level
// after level (the middle, the quartiles, ...), and only the last four probes go to the row itself.  Rows are filled up
// to a multiple of sixteen with the top.  No threshold is above u = 2^32 - 1, so that draw leaves the tree at its last
// leaf, behind the row's end unless M fills the tree: sample_block keeps the probes in the row's last block (`last`
// decides what is drawn).  The index arithmetic is in netmax_search.h.
constexpr int kSampleThreads = 256;

template <int kSampleRows>
__global__ void __launch_bounds__(kSampleThreads) sample_rows_kernel(const SampleParams p, const uint32_t rounds_per_cta) {
  extern __shared__ __align__(16) uint32_t s_thr[];
  const uint32_t M = (uint32_t)p.M, stride = sample_stride(M, kSampleRows), h = sample_levels(M), tree_stride = sample_tree(M, kSampleRows);
  uint32_t* s_tree = s_thr + kSampleRows * stride;
  const uint32_t i0 = blockIdx.x * kSampleRows;
  const uint32_t rows = min((uint32_t)kSampleRows, M - i0);
  for (uint32_t w = 0; w < rows; ++w) {
    const uint32_t* src = p.thresholds + (size_t)(i0 + w) * M;
    uint32_t* dst = s_thr + w * stride;
    if ((M & 3u) == 0u) {
      for (uint32_t j = 4u * threadIdx.x; j < M; j += 4u * kSampleThreads) cp_async_16_stream(dst + j, src + j);
    } else {
#pragma unroll 8
      for (uint32_t j = threadIdx.x; j < M; j += kSampleThreads) dst[j] = __ldg(src + j);
    }
    for (uint32_t j = M + threadIdx.x; j < ((M + 15u) & ~15u); j += kSampleThreads) dst[j] = 0xFFFFFFFFu;
  }
  cp_async_wait_all();
  __syncthreads();
  for (uint32_t e = threadIdx.x; e < rows << h; e += kSampleThreads) {
    const uint32_t w = e >> h, j = e & ((1u << h) - 1u);  // the last threshold before block j -> node
    if (j == 0) continue;
    s_tree[w * tree_stride + sample_node(j, h, __ffs(j) - 1)] = 16u * j <= M ? s_thr[w * stride + 16u * j - 1u] : 0xFFFFFFFFu;
  }
  __syncthreads();
  const uint32_t w = threadIdx.x & (kSampleRows - 1);
  if (w >= rows) return;
  const uint32_t i = i0 + w;
  const uint32_t *row = s_thr + w * stride, *tree = s_tree + w * tree_stride;
  const int32_t last = __ldg(p.last_nz + i);
  const uint32_t begin = blockIdx.y * rounds_per_cta, end = min((uint32_t)p.n_rounds, begin + rounds_per_cta);
  constexpr uint32_t kPerPass = kSampleThreads / kSampleRows;
  constexpr int kAtOnce = 4;  // draws of a thread in flight: a probe's latency is what a single one waits for
  for (uint32_t r = begin + threadIdx.x / kSampleRows; r < end; r += kAtOnce * kPerPass) {
    uint32_t u[kAtOnce], at[kAtOnce];
#pragma unroll
    for (int a = 0; a < kAtOnce; ++a) {
      u[a] = peer_word(p, i, p.first_round + r + a * kPerPass);
      at[a] = 1;
    }
    for (uint32_t l = 0; l < h; ++l) {
#pragma unroll
      for (int a = 0; a < kAtOnce; ++a) at[a] = 2u * at[a] + (tree[at[a]] <= u[a] ? 1u : 0u);
    }
#pragma unroll
    for (int a = 0; a < kAtOnce; ++a) at[a] = 16u * sample_block(at[a], h, M);  // thresholds of whole blocks <= u
#pragma unroll
    for (int s = 8; s > 0; s >>= 1) {
#pragma unroll
      for (int a = 0; a < kAtOnce; ++a)
        if (row[at[a] + s - 1] <= u[a]) at[a] += s;
    }
#pragma unroll
    for (int a = 0; a < kAtOnce; ++a)
      if (r + a * kPerPass < end) put_draw(p, r + a * kPerPass, i, min((int32_t)at[a], last));
  }
}

// ------------------------------------------------------------------------- telemetry
// tel[slot of round k] = (sum over tiles of partials[k][tile]) / M, one warp per round, tiles in a fixed order.
__global__ void __launch_bounds__(256) sum_tile_partials_kernel(const double* partials, int64_t n_tiles, int32_t n_rounds,
                                                                double inv_M, double* tel, int64_t slot0, int64_t ring) {
  const int lane = threadIdx.x & 31;
  const int k = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (k >= n_rounds) return;
  double a = 0.0, b = 0.0;
  for (int64_t t = lane; t < n_tiles; t += 32) {
    a += partials[((size_t)k * n_tiles + t) * 2];
    b += partials[((size_t)k * n_tiles + t) * 2 + 1];
  }
  for (int off = 16; off > 0; off >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, off);
    b += __shfl_down_sync(0xffffffffu, b, off);
  }
  if (lane == 0) {
    double* out = tel + 2 * ((slot0 + k) % ring);
    out[0] = a * inv_M;
    out[1] = b * inv_M;
  }
}

// tel[slot of round k] = sum over chunks of chunk_tel[chunk][slot], chunks in order (a pipelined host
// round trip runs the rounds chunk of columns by chunk; both statistics are sums over columns).
__global__ void __launch_bounds__(256) sum_chunk_telemetry_kernel(const double* chunk_tel, int32_t n_chunks, int64_t ring,
                                                                  int64_t slot0, int64_t n_rounds, double* tel) {
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n_rounds) return;
  const int64_t slot = (slot0 + k) % ring;
  double a = 0.0, b = 0.0;
  for (int c = 0; c < n_chunks; ++c) {
    a += chunk_tel[((size_t)c * ring + slot) * 2];
    b += chunk_tel[((size_t)c * ring + slot) * 2 + 1];
  }
  tel[2 * slot] = a;
  tel[2 * slot + 1] = b;
}

// ------------------------------------------------------------------------- init / IO
struct InitParams {
  float4* dst;  // [M][ldq] column groups
  int64_t ldq, nq;
  int32_t M, tail;  // tail = d % (4 kHalves)
  float stddev;
  uint32_t tag;
  uint32_t q_offset;
  PhiloxKeys keys;
};

template <int kHalves>
__global__ void __launch_bounds__(256) init_normal_kernel(const InitParams p) {
  const int64_t total = (int64_t)p.M * p.nq;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx / p.nq, q = idx - i * p.nq;
    const bool ragged = p.tail != 0 && q == p.nq - 1;
    ulonglong2 o;
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      float4 z = normals4(philox4x32_10((uint32_t)q * kHalves + h + p.q_offset, (uint32_t)i, 0u, p.tag, p.keys));
      z.x *= p.stddev; z.y *= p.stddev; z.z *= p.stddev; z.w *= p.stddev;
      const int live = live_lanes(ragged, p.tail, h);
      if (live < 1) z.x = 0.f;
      if (live < 2) z.y = 0.f;
      if (live < 3) z.z = 0.f;
      if (live < 4) z.w = 0.f;
      const ulonglong2 v = make_ulonglong2(pack2(z.x, z.y), pack2(z.z, z.w));
      if (kHalves == 1) o = v;
      else if (h == 0) o.x = narrow_bf16x4(v);
      else o.y = narrow_bf16x4(v);
    }
    *reinterpret_cast<ulonglong2*>(p.dst + (size_t)i * p.ldq + q) = o;
  }
}

// One stored element as fp32 (bfloat16 widens exactly).
__device__ __forceinline__ float load_element(const void* plane, size_t index, bool bf16) {
  if (bf16) return __uint_as_float((uint32_t)reinterpret_cast<const unsigned short*>(plane)[index] << 16);
  return reinterpret_cast<const float*>(plane)[index];
}

__global__ void __launch_bounds__(256) gather_columns_kernel(const void* x, bool bf16, int64_t ld, int32_t M,
                                                             const int64_t* cols, int64_t n_cols, float* out) {
  const int64_t total = (int64_t)M * n_cols;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx / n_cols, k = idx - i * n_cols;
    out[idx] = load_element(x, (size_t)i * ld + cols[k], bf16);
  }
}

// bfloat16 state <-> dense fp32 rows (host transfers of a bfloat16 context are staged in fp32
// on the device): `rows` rows of d elements; the bfloat16 side has row stride ld.
__global__ void __launch_bounds__(256) narrow_rows_kernel(const float* src, unsigned short* dst, int64_t rows, int64_t d,
                                                          int64_t ld) {
  const int64_t total = rows * d;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx / d, e = idx - i * d;
    unsigned short v;
    asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(v) : "f"(src[idx]));
    dst[(size_t)i * ld + e] = v;
  }
}

__global__ void __launch_bounds__(256) widen_rows_kernel(const unsigned short* src, float* dst, int64_t rows, int64_t d,
                                                         int64_t ld) {
  const int64_t total = rows * d;
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = idx / d, e = idx - i * d;
    dst[idx] = __uint_as_float((uint32_t)src[(size_t)i * ld + e] << 16);
  }
}

}  // namespace netmax
