// CUDA kernels of the NetMax round simulator (sm_100a).
//
//   round_kernel          Eq. 15 (local SGD step with inline Gaussian gradient noise) fused
//                         with Eq. 16 (pull from the round-start snapshot of the peer) and
//                         with the round's telemetry; reads one buffer, writes the other.
//   fused_rounds_kernel   the same for many rounds per launch on tiles that stay in a CTA's shared
//                         memory, a column per thread (long vectors, up to 36 workers).
//   tile_rounds_kernel    (netmax_tiles.cuh) the same with the rows of a tile shared out over the
//                         threads: more workers, and short vectors.
//   pipe_rounds_kernel    (netmax_pipe.cuh) small problems: a warp moves all rows of a few column groups, others
//                         draw its noise and add up its telemetry.
//   multi_round_kernel    short vectors of more workers than fit on chip: all rounds in one launch.
//   step_kernel           the asynchronous timeline: one worker per global step (Eq. 17);
//                         step_tiles_kernel: many steps per launch on resident columns.
// Peer draws, initial state, read-back and sums of telemetry: netmax_plain.cuh.
//
// State precision.  The replicas and centres are stored as fp32 (kHalves == 1) or, as an option
// the paper does not have, as bfloat16 (kHalves == 2).  Either way a thread moves 16-byte column
// groups -- 4 fp32 or 8 bfloat16 values, i.e. kHalves Philox blocks of four normals -- and all
// arithmetic is fp32: bfloat16 values are widened exactly on load, and each new parameter is
// rounded once, to the nearest bfloat16 (ties to even), at the store.
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>

#include "netmax_rng.cuh"

namespace netmax {

// 16 bytes from global to shared memory without passing through registers or L1 (data that no other
// thread of the SM will ask for); completion is awaited by the same thread with cp_async_wait_all.
__device__ __forceinline__ void cp_async_16_stream(void* smem_dst, const void* gmem_src) {
  const uint32_t dst = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(gmem_src) : "memory");
}
// The same for 8 bytes (four bfloat16 values; copies below 16 bytes go through L1).
__device__ __forceinline__ void cp_async_8(void* smem_dst, const void* gmem_src) {
  const uint32_t dst = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Programmatic dependent launch: the sampler lets the kernel behind it start at once; that kernel waits here for the
// sampler to end and its writes to be visible (no-ops where a launch does not ask for it).
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------------- round
struct RoundParams {
  const float4* x_cur;   // [M][ldq] round-start replicas (16-byte column groups: 4 fp32 or 8 bfloat16)
  float4* x_nxt;         // [M][ldq] next replicas
  char* mirror;          // copy of x_nxt in page-locked host memory (short-vector kernel only); may be NULL
  const float4* c;       // [M][ldq] centres
  const int32_t* peers;  // [M] this round's draws
  const float* wtab;     // [M][M] pull weights w_im (fp32)
  double* partials;      // [gridDim.x][2] per-CTA telemetry sums
  unsigned int* ticket;  // last-CTA-done counter (0 between launches)
  double* tel_out;       // [2] this round's (consensus, loss)
  int64_t ldq;           // row stride, in column groups
  uint32_t row_bytes;    // row stride, in bytes (< 2^32)
  int64_t nq;            // column groups per row = ceil(d / (4 kHalves))
  int64_t n_tiles;       // ceil(nq / cg)
  int32_t M;
  int32_t tail;          // d % (4 kHalves): live lanes of the last column group (0 = all of them)
  int32_t cg;            // column groups per tile   (cg * rl == blockDim.x, both powers of two)
  int32_t rl;            // row lanes per tile
  int32_t rg;            // row groups: tile t covers column tile t / rg, rows of group t % rg
  int32_t rows_per_group;  // ceil(M / rg)
  float4* colpart;       // rg > 1: per tile, per column group, per half: (sum, sum of squares) partials
  unsigned int* coltick; // rg > 1: arrivals per column tile (0 between launches)
  float alpha, sigma;    // sigma: the noise scale sigma sqrt(2 ln 2) (see scaled_pair)
  float inv_M;
  uint32_t round_lo, ctr3;
  uint32_t q_offset;     // Philox block index (element / 4) of the context's first element in the global vector
  PhiloxKeys keys;
};

// Per-thread telemetry accumulators.  ColAcc: four columns as two fp32 pairs, sum (x - pivot)
// and sum (x - pivot)^2 over the rows the thread has seen.  LossAcc: sum (x - c)^2 over all of
// the thread's elements.
struct ColAcc {
  pair_t s1a = 0ull, s1b = 0ull, s2a = 0ull, s2b = 0ull;  // +0.0f pairs
};
struct LossAcc {
  pair_t la = 0ull, lb = 0ull;
};

// Four bfloat16 values in a 64-bit word (element 0 in the lowest 16 bits) <-> two fp32 pairs.
// Widening is exact; narrowing rounds to nearest, ties to even.
__device__ __forceinline__ ulonglong2 widen_bf16x4(unsigned long long v) {
  const uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32);
  return make_ulonglong2(pack2(__uint_as_float(lo << 16), __uint_as_float(lo & 0xFFFF0000u)),
                         pack2(__uint_as_float(hi << 16), __uint_as_float(hi & 0xFFFF0000u)));
}
__device__ __forceinline__ unsigned long long narrow_bf16x4(ulonglong2 v) {
  float e0, e1, e2, e3;
  unpack2(v.x, e0, e1);
  unpack2(v.y, e2, e3);
  uint32_t lo, hi;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(e1), "f"(e0));  // first operand -> upper half
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(e3), "f"(e2));
  return ((unsigned long long)hi << 32) | lo;
}
// Half h (four elements, as two fp32 pairs) of a 16-byte column group.
template <int kHalves>
__device__ __forceinline__ ulonglong2 group_half(ulonglong2 raw, int h) {
  if (kHalves == 1) return raw;
  return widen_bf16x4(h == 0 ? raw.x : raw.y);
}
// Live lanes of half h of a column group: 4 everywhere but in a row's last, ragged group.
__device__ __forceinline__ int live_lanes(bool ragged, int tail, int h) {
  return ragged ? min(4, max(0, tail - 4 * h)) : 4;
}

// Eq. 15 and Eq. 16 on one column group of one worker, on packed fp32 pairs:
//   g = (x - c) + n,      h = x - alpha g                                          (Eq. 15)
//   x' = h - w (h - x_m),   w = alpha rho gamma_im  (w = 0 on a self-draw)          (Eq. 16)
// n is sigma times the normals (scaled_normals4; +0 on padding lanes of a row's last, ragged group, which
// hold x = c = 0 and so stay at exactly +0).  ta, tb return x - c for the caller's loss statistic.
// Operand counts matter here: a packed instruction with three distinct register pairs issues every 3.2
// cycles, one with two every 2.2 -- hence subtractions instead of multiply-adds with -1, and the product
// with alpha as scalar multiply-adds that take alpha from the constant bank, except where a kernel is faster with fewer
// instructions (kPairs).
template <int kObjective, int kForm>
__device__ __forceinline__ ulonglong2 update_core(float alpha, ulonglong2 n, ulonglong2 xv, ulonglong2 cv, ulonglong2 xm, float w,
                                                  pair_t& ta, pair_t& tb) {
  ta = sub2(xv.x, cv.x);
  tb = sub2(xv.y, cv.y);
  pair_t ha = xv.x, hb = xv.y;
  if (kObjective == 1 && (kForm & kPairs)) {
    const pair_t nalpha2 = pack2(-alpha, -alpha);
    ha = fma2(nalpha2, add2(ta, n.x), xv.x);
    hb = fma2(nalpha2, add2(tb, n.y), xv.y);
  } else if (kObjective == 1) {
    float g0, g1, g2, g3, x0, x1, x2, x3;
    unpack2(add2(ta, n.x), g0, g1);
    unpack2(add2(tb, n.y), g2, g3);
    unpack2(xv.x, x0, x1);
    unpack2(xv.y, x2, x3);
    ha = pack2(fmaf(-alpha, g0, x0), fmaf(-alpha, g1, x1));
    hb = pack2(fmaf(-alpha, g2, x2), fmaf(-alpha, g3, x3));
  }
  const pair_t nw2 = pack2(-w, -w);
  return make_ulonglong2(fma2(nw2, sub2(ha, xm.x), ha), fma2(nw2, sub2(hb, xm.y), hb));
}

// The noise of one column group of one worker, with its Philox block drawn on the spot.
template <int kObjective, int kForm>
__device__ __forceinline__ ulonglong2 draw_noise(float sigma_s, const PhiloxKeys& keys, uint32_t iter_lo, uint32_t ctr3, uint32_t q32,
                                                 uint32_t worker, int live) {
  if (kObjective != 1) return make_ulonglong2(0ull, 0ull);
  const ulonglong2 n = scaled_normals4<kForm>(philox4x32_10(q32, worker, iter_lo, ctr3, keys), sigma_s);
  return live < 4 ? mask_lanes(n, live) : n;
}

// update_core plus the telemetry sums of the round-start values.  kObjective == 2 measures only.
template <int kObjective, int kForm>
__device__ __forceinline__ ulonglong2 row_update(float alpha, ulonglong2 n, ulonglong2 xv, ulonglong2 cv, ulonglong2 xm,
                                                 ulonglong2 pivot, float w, ColAcc& acc, LossAcc& lacc) {
  pair_t ta, tb;
  ulonglong2 o = xv;
  if (kObjective == 2) {
    ta = sub2(xv.x, cv.x);
    tb = sub2(xv.y, cv.y);
  } else {
    o = update_core<kObjective, kForm>(alpha, n, xv, cv, xm, w, ta, tb);
  }
  const pair_t da = sub2(xv.x, pivot.x), db = sub2(xv.y, pivot.y);
  acc.s1a = add2(acc.s1a, da);
  acc.s1b = add2(acc.s1b, db);
  acc.s2a = fma2(da, da, acc.s2a);
  acc.s2b = fma2(db, db, acc.s2b);
  lacc.la = fma2(ta, ta, lacc.la);
  lacc.lb = fma2(tb, tb, lacc.lb);
  return o;
}

// Block reduction of a CTA's two telemetry sums into partials[2 * blockIdx.x ..].
// s_red: 64 doubles of shared memory.  Every thread of the CTA must call this.
__device__ __forceinline__ void block_partials(double* partials, double acc_cons, double acc_loss, double* s_red) {
  const int tid = threadIdx.x;
  acc_loss *= 0.5;
  for (int off = 16; off > 0; off >>= 1) {
    acc_cons += __shfl_down_sync(0xffffffffu, acc_cons, off);
    acc_loss += __shfl_down_sync(0xffffffffu, acc_loss, off);
  }
  const int warp = tid >> 5, lane = tid & 31, nwarps = blockDim.x >> 5;
  __syncthreads();  // s_red may still be read by an earlier call
  if (lane == 0) {
    s_red[warp] = acc_cons;
    s_red[32 + warp] = acc_loss;
  }
  __syncthreads();
  if (tid == 0) {
    double a = 0.0, b = 0.0;
    for (int wi = 0; wi < nwarps; ++wi) {
      a += s_red[wi];
      b += s_red[32 + wi];
    }
    partials[2 * (size_t)blockIdx.x] = a;
    partials[2 * (size_t)blockIdx.x + 1] = b;
  }
}

// Adds all CTA partials in index order (deterministic) and writes the round's telemetry.
// Every thread of the (one) calling CTA must call this.
__device__ __forceinline__ void sum_partials(const double* partials, double inv_M, double* tel_out, double* s_red) {
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31, nwarps = blockDim.x >> 5;
  double a = 0.0, b = 0.0;
  for (unsigned int j = tid; j < gridDim.x; j += blockDim.x) {
    a += __ldcg(partials + 2 * (size_t)j);
    b += __ldcg(partials + 2 * (size_t)j + 1);
  }
  for (int off = 16; off > 0; off >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, off);
    b += __shfl_down_sync(0xffffffffu, b, off);
  }
  __syncthreads();
  if (lane == 0) {
    s_red[warp] = a;
    s_red[32 + warp] = b;
  }
  __syncthreads();
  if (tid == 0) {
    a = 0.0;
    b = 0.0;
    for (int wi = 0; wi < nwarps; ++wi) {
      a += s_red[wi];
      b += s_red[32 + wi];
    }
    tel_out[0] = a * inv_M;
    tel_out[1] = b * inv_M;
  }
}

// One launch per round: the last CTA of the grid to publish its partials sums them.
__device__ __forceinline__ void finalize_telemetry(const RoundParams& p, double acc_cons, double acc_loss, double* s_red) {
  block_partials(p.partials, acc_cons, acc_loss, s_red);
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned int t = atomicAdd(p.ticket, 1u);
    s_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    sum_partials(p.partials, (double)p.inv_M, p.tel_out, s_red);
    if (threadIdx.x == 0) *p.ticket = 0u;
  }
}

// A launch of several rounds: the last CTA of the grid to publish its partials [n_rounds][gridDim.x][2] adds
// them, a warp per round, in a fixed order.  Every thread must call this.
__device__ __forceinline__ void finalize_rounds(const double* partials, int n_rounds, double inv_M, double* tel, int64_t slot0,
                                                int64_t ring, unsigned int* ticket) {
  __shared__ bool s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int lane = threadIdx.x & 31;
  for (int k = threadIdx.x >> 5; k < n_rounds; k += blockDim.x >> 5) {
    double a = 0.0, b = 0.0;
    for (unsigned int j = lane; j < gridDim.x; j += 32) {
      const double2 v = __ldcg(reinterpret_cast<const double2*>(partials) + (size_t)k * gridDim.x + j);
      a += v.x;
      b += v.y;
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
  if (threadIdx.x == 0) *ticket = 0u;
}

// Direct-load round kernel (any M).  One tile = all M rows (or, for short vectors with many
// workers, one of rg row groups) x cg column groups.  Thread (cgi, rli) owns column group cgi
// of the tile and the rows rli, rli + rl, ... of its row group; tiles are taken round-robin by
// the resident CTAs.  All accesses are plain cacheable 128-bit loads and
// stores: the peer read (a row this tile reads anyway) then hits L1/L2, and streaming hints on
// c and on the output measured slower.
// Dynamic shared memory: (peer, weight) int2[M], then (rl > 1) 2 * kHalves * blockDim float4 of
// column-sum scratch, then 64 doubles for the block reduction.
#ifndef NETMAX_ROUND_MIN_CTAS
#define NETMAX_ROUND_MIN_CTAS 4  // CTAs per SM the register allocation leaves room for
#endif
#ifndef NETMAX_ROUND_MIN_CTAS_BF16
#define NETMAX_ROUND_MIN_CTAS_BF16 2  // bfloat16 state: eight elements per thread; measured 152 us (2), 161 (3), 157 (4) per cfg2 round
#endif

// kRowsInFlight = 1 (64 registers, 4 CTAs/SM) is the streaming shape for long vectors, where
// occupancy hides the HBM latency; kRowsInFlight = 4 (2 CTAs/SM) serves short, L2-resident
// problems, where a thread's chain of dependent row loads is what takes the time.
// this round's (peer, weight) of workers [r0, r1) into shared memory
__device__ __forceinline__ void load_draws(const RoundParams& p, const int32_t* peers, int2* s_pw, int r0, int r1) {
  for (int i = r0 + threadIdx.x; i < r1; i += blockDim.x) {
    const int32_t m = __ldg(peers + i);
    s_pw[i] = make_int2(m, __float_as_int((m == i) ? 0.0f : __ldg(p.wtab + (size_t)i * p.M + m)));
  }
}

// Loads of replica data.  Inside one launch per round the round-start buffer is read-only
// (non-coherent path); a launch that runs several rounds reads what other SMs wrote a round
// earlier and must bypass L1.
template <bool kCoherent>
__device__ __forceinline__ ulonglong2 ld_x(const char* ptr) {
  return kCoherent ? __ldcg(reinterpret_cast<const ulonglong2*>(ptr)) : __ldg(reinterpret_cast<const ulonglong2*>(ptr));
}

// All tiles of this CTA for one round.  Every thread of the CTA must call this.
template <int kObjective, int kRowsInFlight, bool kCoherent, int kHalves>
__device__ __forceinline__ void round_tiles(const RoundParams& p, const float4* x_cur, float4* x_nxt, const int32_t* peers,
                                            uint32_t round_lo, uint32_t ctr3, int2* s_pw, float4* s_col,
                                            double& acc_cons, double& acc_loss) {
  constexpr int kStats = 2 * kHalves;  // float4 column statistics per thread: (sum, sum of squares) per half
  const int tid = threadIdx.x;
  const int G = p.rg;
  __shared__ bool s_lastcol;
  const int cgi = tid & (p.cg - 1);
  const int rli = tid / p.cg;
  const int M = p.M;
  const int step = p.rl;
  if (G == 1 && kObjective != 2) {
    __syncthreads();  // readers of the previous round's draws are done
    load_draws(p, peers, s_pw, 0, M);
    __syncthreads();
  }

  for (int64_t tile = blockIdx.x; tile < p.n_tiles; tile += gridDim.x) {
    const int64_t ct = G == 1 ? tile : tile / G;      // column tile
    const int grp = G == 1 ? 0 : (int)(tile - ct * G);  // row group
    const int r0 = grp * p.rows_per_group, r1 = min(M, r0 + p.rows_per_group);
    if (G > 1 && kObjective != 2) {
      __syncthreads();  // the previous tile's readers of s_pw are done
      load_draws(p, peers, s_pw, r0, r1);
      __syncthreads();
    }
    const int64_t q = ct * p.cg + cgi;
    const bool live = q < p.nq;
    const bool ragged = (p.tail != 0) && (q == p.nq - 1);
    float4 st[kStats];  // st[2h] = sum (x - pivot), st[2h + 1] = sum (x - pivot)^2 of half h's columns
#pragma unroll
    for (int a = 0; a < kStats; ++a) st[a] = make_float4(0.f, 0.f, 0.f, 0.f);
    float loss = 0.f;
    if (live) {
      // byte pointers to this thread's column group in row 0; row i is i * row_bytes further
      const char* xq = reinterpret_cast<const char*>(x_cur + q);
      const char* cq = reinterpret_cast<const char*>(p.c + q);
      char* oq = reinterpret_cast<char*>(x_nxt + q);
      const uint32_t q32 = (uint32_t)q * kHalves + p.q_offset;
      const ulonglong2 pivot = ld_x<kCoherent>(xq);  // row 0: pivot of the one-pass variance
      ColAcc acc[kHalves];
      LossAcc lacc;
      for (int i0 = r0 + rli; i0 < r1; i0 += step * kRowsInFlight) {
        ulonglong2 xv[kRowsInFlight], xm[kRowsInFlight], cv[kRowsInFlight];
        int2 pw[kRowsInFlight];
#pragma unroll
        for (int u = 0; u < kRowsInFlight; ++u) {  // issue the loads of kRowsInFlight rows
          const int i = i0 + u * step;
          if (kRowsInFlight == 1 || i < r1) {
            const uint64_t row = (uint64_t)(uint32_t)i * p.row_bytes;
            xv[u] = ld_x<kCoherent>(xq + row);
            if (kObjective == 2) {  // measuring: no peers involved
              pw[u] = make_int2(i, 0);
              xm[u] = xv[u];
            } else {
              pw[u] = s_pw[i];
              xm[u] = ld_x<kCoherent>(xq + (uint64_t)(uint32_t)pw[u].x * p.row_bytes);
            }
            cv[u] = __ldg(reinterpret_cast<const ulonglong2*>(cq + row));
          }
        }
#pragma unroll
        for (int u = 0; u < kRowsInFlight; ++u) {
          const int i = i0 + u * step;
          if (kRowsInFlight == 1 || i < r1) {
            ulonglong2 o;
#pragma unroll
            for (int h = 0; h < kHalves; ++h) {
              // (the mantissa by shift and or: 8 x 8,388,611 elements 154.2 us per round, with the funnel shift 159.9; padding
              // lanes cleared behind the update: a test between the noise and the update keeps their instructions apart, 157.0)
              const ulonglong2 noise = draw_noise<kObjective, 0>(p.sigma, p.keys, round_lo, ctr3, q32 + h, (uint32_t)i, 4);
              ulonglong2 oh = row_update<kObjective, 0>(p.alpha, noise, group_half<kHalves>(xv[u], h), group_half<kHalves>(cv[u], h),
                                                        group_half<kHalves>(xm[u], h), group_half<kHalves>(pivot, h),
                                                        __int_as_float(pw[u].y), acc[h], lacc);
              const int live = live_lanes(ragged, p.tail, h);
              if (live < 4) oh = mask_lanes(oh, live);
              if (kHalves == 1) o = oh;
              else if (h == 0) o.x = narrow_bf16x4(oh);
              else o.y = narrow_bf16x4(oh);
            }
            if (kObjective != 2) *reinterpret_cast<ulonglong2*>(oq + (uint64_t)(uint32_t)i * p.row_bytes) = o;
            if (kRowsInFlight != 1 && !kCoherent && kObjective != 2 && p.mirror)
              *reinterpret_cast<ulonglong2*>(p.mirror + (uint64_t)q * 16u + (uint64_t)(uint32_t)i * p.row_bytes) = o;
          }
        }
      }
#pragma unroll
      for (int h = 0; h < kHalves; ++h) {
        unpack2(acc[h].s1a, st[2 * h].x, st[2 * h].y);
        unpack2(acc[h].s1b, st[2 * h].z, st[2 * h].w);
        unpack2(acc[h].s2a, st[2 * h + 1].x, st[2 * h + 1].y);
        unpack2(acc[h].s2b, st[2 * h + 1].z, st[2 * h + 1].w);
      }
      float l0, l1, l2, l3;
      unpack2(lacc.la, l0, l1);
      unpack2(lacc.lb, l2, l3);
      loss = (l0 + l1) + (l2 + l3);
    }
    if (p.rl > 1) {  // sum the column statistics over the row lanes (stride cg in tid)
#pragma unroll
      for (int a = 0; a < kStats; ++a) s_col[a * blockDim.x + tid] = st[a];
      __syncthreads();
      for (int s = blockDim.x >> 1; s >= p.cg; s >>= 1) {
        if (tid < s) {
#pragma unroll
          for (int a = 0; a < kStats; ++a) {
            float4 v = s_col[a * blockDim.x + tid];
            const float4 b = s_col[a * blockDim.x + tid + s];
            v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w;
            s_col[a * blockDim.x + tid] = v;
          }
        }
        __syncthreads();
      }
#pragma unroll
      for (int a = 0; a < kStats; ++a) st[a] = s_col[a * blockDim.x + cgi];
      __syncthreads();
    }
    bool owner = true;  // does this CTA hold the complete column sums of the tile?
    if (G > 1) {
      // rows are split over rg CTAs: publish this CTA's column partials; the last of the rg
      // CTAs of a column tile to arrive adds them up in group order (deterministic)
      if (rli == 0) {
#pragma unroll
        for (int a = 0; a < kStats; ++a) p.colpart[((size_t)tile * p.cg + cgi) * kStats + a] = st[a];
      }
      __threadfence();
      __syncthreads();
      if (tid == 0) {
        const unsigned int t = atomicAdd(p.coltick + ct, 1u);
        s_lastcol = (t == (unsigned int)G - 1);
        if (s_lastcol) p.coltick[ct] = 0u;
      }
      __syncthreads();
      owner = s_lastcol;
      if (owner && rli == 0) {
        __threadfence();
#pragma unroll
        for (int a = 0; a < kStats; ++a) st[a] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int gg = 0; gg < G; ++gg) {
#pragma unroll
          for (int a = 0; a < kStats; ++a) {
            const float4 b = __ldcg(p.colpart + (((size_t)ct * G + gg) * p.cg + cgi) * kStats + a);
            st[a].x += b.x; st[a].y += b.y; st[a].z += b.z; st[a].w += b.w;
          }
        }
      }
    }
    if (rli == 0 && owner) {
      // sum_i (x_i - xbar)^2 = sum_i (x_i - a)^2 - (sum_i (x_i - a))^2 / M   per column
#pragma unroll
      for (int h = 0; h < kHalves; ++h) {
        const float4 s1 = st[2 * h], s2 = st[2 * h + 1];
        const float cons = (s2.x - s1.x * s1.x * p.inv_M) + (s2.y - s1.y * s1.y * p.inv_M) +
                           (s2.z - s1.z * s1.z * p.inv_M) + (s2.w - s1.w * s1.w * p.inv_M);
        acc_cons += (double)cons;
      }
    }
    acc_loss += (double)loss;
  }
}

// kRowsInFlight = 1 (64 registers, 4 CTAs/SM) is the streaming shape for long vectors, where
// occupancy hides the HBM latency; kRowsInFlight = 4 (2 CTAs/SM) serves short, L2-resident
// problems, where a thread's chain of dependent row loads is what takes the time.
template <int kObjective, int kRowsInFlight, int kHalves>
__global__ void __launch_bounds__(256, kRowsInFlight != 1 ? 2 : kHalves == 1 ? NETMAX_ROUND_MIN_CTAS : NETMAX_ROUND_MIN_CTAS_BF16)
    round_kernel(const RoundParams p) {
  if (kRowsInFlight != 1) wait_for_previous();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  int2* s_pw = reinterpret_cast<int2*>(smem_raw);  // (peer, bits of the pull weight) per worker
  const size_t head = (((size_t)p.M * 8) + 15) & ~(size_t)15;
  float4* s_col = reinterpret_cast<float4*>(smem_raw + head);
  double* s_red = reinterpret_cast<double*>(smem_raw + head + (p.rl > 1 ? (size_t)blockDim.x * 32 * kHalves : 0));
  double acc_cons = 0.0, acc_loss = 0.0;
  round_tiles<kObjective, kRowsInFlight, false, kHalves>(p, p.x_cur, p.x_nxt, p.peers, p.round_lo, p.ctr3, s_pw,
                                                                     s_col, acc_cons, acc_loss);
  finalize_telemetry(p, acc_cons, acc_loss, s_red);
}

// ---- several rounds in one launch (short, L2-resident problems) ------------------------------
// For problems of a few microseconds per round the launch and the chain of dependent global
// round trips are what take the time.  This kernel is launched cooperatively (all CTAs
// resident), runs n_rounds rounds back to back and separates them with a grid-wide barrier: an
// arrival counter in global memory that every CTA polls a bounded number of times.  A CTA
// whose wait runs out raises *error and leaves; the others then run out as well.
struct MultiRoundParams {
  RoundParams r;          // x_cur / x_nxt: the buffers of the first round; peers, tel_out, round_lo, ctr3 unused
  const int32_t* trace;   // peer-trace ring [ring][M], filled for these rounds by sample_peers_kernel
  double* tel;            // telemetry ring [ring][2]
  double* partials2;      // [2][gridDim.x][2]: CTA partials, alternating by round
  unsigned int* barrier;  // arrival counter, 0 at launch
  unsigned int* error;    // raised when a barrier wait gave up
  int64_t slot0, ring;    // ring slot of the first round
  uint64_t first_round;
  int32_t n_rounds;
  uint32_t absent_ctas;   // test hook: the barrier also waits for this many CTAs that do not exist
};

constexpr uint32_t kBarrierSpinLimit = 1u << 21;

// Grid-wide barrier number `epoch` (1, 2, ...).  Returns false if the wait gave up.
__device__ __forceinline__ bool grid_barrier(unsigned int* counter, unsigned int epoch, unsigned int* error,
                                             unsigned int absent_ctas) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();  // this CTA's writes of the round are visible before it is counted
    atomicAdd(counter, 1u);
    const unsigned int target = epoch * (gridDim.x + absent_ctas);
    int ok = 0;
    for (uint32_t it = 0; it < kBarrierSpinLimit; ++it) {
      if (*reinterpret_cast<volatile unsigned int*>(counter) >= target) {
        ok = 1;
        break;
      }
      __nanosleep(32);
    }
    if (!ok) *reinterpret_cast<volatile unsigned int*>(error) = 1u;  // (page-locked host memory)
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

template <int kObjective, int kHalves>
__global__ void __launch_bounds__(256, 2) multi_round_kernel(const MultiRoundParams mp) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const RoundParams& p = mp.r;
  int2* s_pw = reinterpret_cast<int2*>(smem_raw);
  const size_t head = (((size_t)p.M * 8) + 15) & ~(size_t)15;
  float4* s_col = reinterpret_cast<float4*>(smem_raw + head);
  double* s_red = reinterpret_cast<double*>(smem_raw + head + (p.rl > 1 ? (size_t)blockDim.x * 32 * kHalves : 0));
  const float4* x_cur = p.x_cur;
  float4* x_nxt = p.x_nxt;
  for (int k = 0; k < mp.n_rounds; ++k) {
    const uint64_t round = mp.first_round + (uint64_t)k;
    const int64_t slot = (mp.slot0 + k) % mp.ring;
    double* partials = mp.partials2 + (size_t)(k & 1) * 2 * gridDim.x;
    double acc_cons = 0.0, acc_loss = 0.0;
    round_tiles<kObjective, 4, true, kHalves>(p, x_cur, x_nxt, mp.trace + slot * p.M, (uint32_t)round,
                                                          philox_ctr3(kTagNoise, round), s_pw, s_col, acc_cons, acc_loss);
    block_partials(partials, acc_cons, acc_loss, s_red);
    if (!grid_barrier(mp.barrier, (unsigned int)(k + 1), mp.error, mp.absent_ctas)) return;
    // round k is complete everywhere: one CTA publishes its telemetry while the rest move on
    // (partials alternate, so round k+1 cannot overwrite what is being summed here)
    if (blockIdx.x == 0) sum_partials(partials, (double)p.inv_M, mp.tel + 2 * slot, s_red);
    const float4* t = x_cur;
    x_cur = x_nxt;
    x_nxt = const_cast<float4*>(t);
  }
}

// ---- several rounds over one resident tile (long vectors, few workers) -----------------------
// Given the peer draws, every column of the M x d state evolves on its own (Eq. 16 is
// elementwise), so a tile that holds ALL M rows of a column range can be advanced several
// rounds without touching global memory in between: the HBM traffic per element drops from
// 12 bytes per round (x and c read, x' written; the peer read is a cache hit) to 12 bytes per
// kFusedMaxRounds rounds, and the kernel becomes bound by its arithmetic instead.
//
// A thread owns one 16-byte column group for all M rows.  Its slab of shared memory
// ([2][M] replica values, double-buffered by round, and [M] centres, each entry 16 bytes,
// laid out [row][thread] so that a warp's accesses are conflict-free) is private to the thread:
// the peer's value of the same column group was written by this very thread a round earlier,
// so the rounds need no barrier.  Per-element arithmetic is row_update's, hence the replicas
// are bit-identical to one launch per round; telemetry sums only differ in the order of their
// double-precision accumulation.  The slabs always hold fp32; with bfloat16 state (kBf16) a
// thread's column group is four bfloat16 values (8 bytes of global memory), widened on the way
// in, and every round's result is rounded to bfloat16 before it is written to the slab, exactly
// as a store to and a load from the bfloat16 state would.
#ifndef NETMAX_FUSED_PREFETCH
#define NETMAX_FUSED_PREFETCH 1  // fetch the next tile under the last round of the current one (fp32 state)
#endif
constexpr int kFusedMaxRounds = 32;  // rounds per launch of fused_rounds_kernel, at most

struct FusedParams {
  const float4* x_cur;   // [M][ldq] replicas at the start of the first round
  float4* x_nxt;         // [M][ldq] replicas after the last round
  const float4* c;       // [M][ldq]
  const int32_t* trace;  // peer-trace ring [ring][M], filled for these rounds
  const float* wtab;     // [M][M]
  double* tel;           // telemetry ring [ring][2]
  double* partials;      // [n_rounds][gridDim.x][2]
  unsigned int* ticket;  // last-CTA-done counter (0 between launches)
  int64_t slot0, ring;   // ring slot of the first round
  uint64_t first_round;  // (its high word is that of all rounds of the launch)
  int32_t n_rounds;      // 1 .. slots
  int32_t slots;         // rounds the table of draws at the head of the shared memory has room for (<= kFusedMaxRounds)
  int64_t nq, n_tiles;   // column groups of FOUR elements per row (whatever the storage), tiles of blockDim of them
  uint32_t row_bytes;
  int32_t M, tail;       // tail = d % 4
  float alpha, sigma, inv_M;
  uint32_t q_offset;
  PhiloxKeys keys;
};

// Dynamic shared memory: (peer row offset, weight) int2[slots][M] -- with kStart (peer row offset, weight, noise_start of the
// row) int4[slots][M] --, the warps' telemetry sums double[slots][warps][2], then the slabs float4[3][M][blockDim] (replicas of even rounds, of odd rounds,
// centres).  Any block size that is a multiple of 32 up to 256 works.
// The telemetry of a round is added over the lanes of a warp at its end (in double) and kept per warp in shared memory,
// for up to 32 rounds; launches of at most kReg rounds keep a thread's own sums in registers instead, which spares a
// round's shuffles (us per call, sums in shared memory / in registers: 2 x 33,554,435 elements, 8 rounds 961 / 916, 4
// rounds 515 / 492; 8 x 8,388,611: 702 / 690, 371 / 367).
// kStart: the first product of a row's noise depends on the worker and the round alone, so a table holds it for all threads;
// column and round parts of the others are worked out once per tile and once per round (noise_column, noise_base).  us per
// launch of 20 rounds, without / with all three: 8 x 11,173,962 elements 2,204 / 2,060, bfloat16 state 2,336 / 2,130, 16 x
// 8,000,002 3,168 / 3,050, 4 x 8,000,002 912 / 843; eight rounds of 2 x 33,554,435 899 / 802.  Above kStartWorkers the wider
// table costs rounds per launch, and the one warp per scheduler gains nothing from it (28 x 2,000,002, 8 rounds: 769 before, 765
// with it, 745 without).  It costs them with twelve workers too, eight instead of sixteen, and gains all the same (12 x 4,000,002, 16 and 64
// rounds, narrow / wide: 1,010 / 978, 3,971 / 3,842; bfloat16 state 1,064 / 1,018, 4,193 / 4,005).
constexpr int kStartWorkers = 17;
__host__ __device__ inline uint32_t fused_draw_bytes(int64_t M) { return M <= kStartWorkers ? 16u : 8u; }
__host__ __device__ inline uint32_t fused_head(int slots, int64_t M, int threads) {
  return (uint32_t)(((uint64_t)slots * (uint64_t)(M * fused_draw_bytes(M) + (threads >> 5) * 16) + 127u) & ~(uint64_t)127u);
}
template <int kObjective, bool kBf16, int kReg, bool kStart>
__global__ void __launch_bounds__(256, 2) fused_rounds_kernel(const FusedParams p) {
  constexpr uint32_t kGroupBytes = kBf16 ? 8u : 16u;  // four elements in global memory
  constexpr int kUnroll = kStart ? 2 : 4;             // rows of a round in flight per thread
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int tid = threadIdx.x, T = blockDim.x, M = p.M;
  using Draw = typename std::conditional<kStart, int4, int2>::type;
  Draw* s_pw = reinterpret_cast<Draw*>(smem_raw);  // (byte offset of the peer's row in a slab, pull weight, start of the noise)
  const uint32_t head = fused_head(p.slots, M, T);
  double* s_tel = reinterpret_cast<double*>(smem_raw + (size_t)p.slots * M * sizeof(Draw));
  const int lane = tid & 31, warp = tid >> 5, nwarps = T >> 5;
  const uint32_t stride = (uint32_t)T * 16u;     // bytes between consecutive rows of a slab
  const uint32_t plane = (uint32_t)M * stride;   // bytes of one [M][T] slab
  unsigned char* slab = smem_raw + head + (uint32_t)tid * 16u;  // this thread's column: slabs 0, 1 (replicas), 2 (centres)

  double acc_cons[kReg > 0 ? kReg : 1], acc_loss[kReg > 0 ? kReg : 1];
#pragma unroll
  for (int k = 0; k < kReg; ++k) acc_cons[k] = acc_loss[k] = 0.0;
  if (kReg == 0)
    for (int k = tid; k < p.n_rounds * nwarps * 2; k += T) s_tel[k] = 0.0;
  for (int k = 0; k < p.n_rounds; ++k) {
    const int32_t* peers = p.trace + ((p.slot0 + k) % p.ring) * M;
    for (int i = tid; i < M; i += T) {
      const int32_t m = __ldg(peers + i);
      Draw d;
      d.x = (int)((uint32_t)m * stride);
      d.y = __float_as_int((m == i) ? 0.0f : __ldg(p.wtab + (size_t)i * M + m));
      if constexpr (kStart) {
        const uint64_t start = noise_start((uint32_t)i, (uint32_t)(p.first_round + (uint64_t)k), p.keys);
        d.z = (int)(uint32_t)start;
        d.w = (int)(uint32_t)(start >> 32);
      }
      s_pw[k * M + i] = d;
    }
  }
  __syncthreads();

  // Slab `base` (0 or 1) holds the tile's values at the start of the first round; round k reads
  // slab (base + k) & 1 and writes the other one.  The LAST round of a tile writes its results
  // straight to global memory, which leaves its would-be output slab idle for that whole round:
  // the next tile's replicas are fetched into it (cp.async, fp32 state), and the next tile's centre
  // of a row replaces the current one as soon as that row has been updated for the last time.  The
  // global loads of a tile thus run under the last round of its predecessor.  Every slab slot is
  // read and written by its own thread only, so cp.async.wait_all is all the synchronisation needed.
  // bfloat16 state arrives as the 8 stored bytes in the low half of a 16-byte slot and is widened in
  // place when the tile starts.
  constexpr bool kPrefetch = NETMAX_FUSED_PREFETCH != 0;
  // (us per call, scalar steps / steps on pairs: fp32, 36 x 1,864,138 elements, 4 rounds 462 / 475, 8 rounds 899 / 880;
  // 8 x 8,388,611 367 / 371, 690 / 681, 20 rounds 1,707 / 1,680; bfloat16 state 387 / 381, 721 / 706; the radius's mantissa
  // by a funnel shift: 1 to 2 % slower throughout)
  constexpr int kForm = kBf16 || kReg != 4 ? kPairs : 0;
  uint32_t base = 0;
  bool fetched = false;  // has this tile been fetched by the previous one?
  for (int64_t tile = blockIdx.x; tile < p.n_tiles; tile += gridDim.x) {
    const int64_t q = tile * T + tid;
    const bool live = q < p.nq;  // (no barrier below: warps are independent)
    const int lanes = live ? live_lanes((p.tail != 0) && (q == p.nq - 1), p.tail, 0) : 0;
    const NoiseColumn column = noise_column((uint32_t)q + p.q_offset, philox_ctr3(kTagNoise, p.first_round), p.keys);
    const int64_t q_next = q + (int64_t)gridDim.x * T;
    const bool have_next = kPrefetch && tile + gridDim.x < p.n_tiles && q_next < p.nq;
    if (fetched) {
      cp_async_wait_all();
      if (kBf16) {
        unsigned char* sx = slab + base * plane;
        unsigned char* sc = slab + 2u * plane;
#pragma unroll 4
        for (int i = 0; i < M; ++i) {
          *reinterpret_cast<ulonglong2*>(sx) = widen_bf16x4(*reinterpret_cast<const unsigned long long*>(sx));
          *reinterpret_cast<ulonglong2*>(sc) = widen_bf16x4(*reinterpret_cast<const unsigned long long*>(sc));
          sx += stride;
          sc += stride;
        }
      }
    } else if (live) {  // all rows of this column group into the thread's slabs
      const char* xq = reinterpret_cast<const char*>(p.x_cur) + (uint64_t)q * kGroupBytes;
      const char* cq = reinterpret_cast<const char*>(p.c) + (uint64_t)q * kGroupBytes;
      unsigned char* sx = slab + base * plane;
      unsigned char* sc = slab + 2u * plane;
#pragma unroll 4
      for (int i = 0; i < M; ++i) {
        if (kBf16) {
          *reinterpret_cast<ulonglong2*>(sx) = widen_bf16x4(__ldg(reinterpret_cast<const unsigned long long*>(xq)));
          *reinterpret_cast<ulonglong2*>(sc) = widen_bf16x4(__ldg(reinterpret_cast<const unsigned long long*>(cq)));
        } else {
          *reinterpret_cast<ulonglong2*>(sx) = __ldg(reinterpret_cast<const ulonglong2*>(xq));
          *reinterpret_cast<ulonglong2*>(sc) = __ldg(reinterpret_cast<const ulonglong2*>(cq));
        }
        xq += p.row_bytes;
        cq += p.row_bytes;
        sx += stride;
        sc += stride;
      }
    }
    unsigned char* const cen = slab + 2u * plane;
    char* const oq = reinterpret_cast<char*>(p.x_nxt) + (uint64_t)q * kGroupBytes;
    const char* const cq_next = reinterpret_cast<const char*>(p.c) + (uint64_t)q_next * kGroupBytes;

    // one round over the thread's column group; kLast: the tile's last round (see above)
    auto run_round = [&](int k, auto last_tag, auto ragged_tag) {
      constexpr bool kLast = decltype(last_tag)::value;
      constexpr bool kRagged = decltype(ragged_tag)::value;
      const unsigned char* cur = slab + ((base + (uint32_t)k) & 1u) * plane;
      unsigned char* nxt = slab + ((base + (uint32_t)k + 1u) & 1u) * plane;
      if (kLast && have_next) {
        const char* xq = reinterpret_cast<const char*>(p.x_cur) + (uint64_t)q_next * kGroupBytes;
        unsigned char* sx = nxt;
#pragma unroll 4
        for (int i = 0; i < M; ++i) {
          if (kBf16) cp_async_8(sx, xq);
          else cp_async_16_stream(sx, xq);
          xq += p.row_bytes;
          sx += stride;
        }
      }
      const Draw* pw = s_pw + k * M;
      const ulonglong2 pivot = *reinterpret_cast<const ulonglong2*>(cur);
      ColAcc acc;
      LossAcc lacc;
      uint32_t off = 0;
      uint64_t goff = 0;
      auto do_row = [&](Draw d, uint4 rnd) {
        if (kRagged && !live) return;
        ulonglong2 noise = kObjective == 1 ? scaled_normals4<kForm>(rnd, p.sigma) : make_ulonglong2(0ull, 0ull);
        if (kRagged) noise = mask_lanes(noise, lanes);
        const ulonglong2 o = row_update<kObjective, kForm>(
            p.alpha, noise, *reinterpret_cast<const ulonglong2*>(cur + off), *reinterpret_cast<const ulonglong2*>(cen + off),
            *reinterpret_cast<const ulonglong2*>(cur + (uint32_t)d.x), pivot, __int_as_float(d.y), acc, lacc);
        if (kLast) {
          if (kBf16) *reinterpret_cast<unsigned long long*>(oq + goff) = narrow_bf16x4(o);
          else *reinterpret_cast<ulonglong2*>(oq + goff) = o;
          if (have_next) {  // this row's centre is not read again in this tile
            if (kBf16) cp_async_8(cen + off, cq_next + goff);
            else cp_async_16_stream(cen + off, cq_next + goff);
          }
          goff += p.row_bytes;
        } else {
          *reinterpret_cast<ulonglong2*>(nxt + off) = kBf16 ? widen_bf16x4(narrow_bf16x4(o)) : o;
        }
        off += stride;
      };
      // the Philox block of row i + 1 is drawn while row i goes through Box-Muller and Eq. 15-16:
      // the two are independent, so the integer multiplies of the one fill the latencies of the other
      const NoiseBase nb = noise_base(column, (uint32_t)(p.first_round + (uint64_t)k), p.keys);
      auto words = [&](int i, Draw d) {
        if constexpr (kStart) return noise_words(nb, (uint32_t)d.z | (uint64_t)(uint32_t)d.w << 32, p.keys);
        else return noise_words(nb, (uint32_t)i, p.keys);
      };
      Draw next = pw[0];
      uint4 rnd = words(0, next);
#pragma unroll kUnroll
      for (int i = 0; i + 1 < M; ++i) {
        const Draw d = next;
        next = pw[i + 1];
        const uint4 rnd_next = words(i + 1, next);
        do_row(d, rnd);
        rnd = rnd_next;
      }
      do_row(next, rnd);
      float4 s1, s2;
      unpack2(acc.s1a, s1.x, s1.y);
      unpack2(acc.s1b, s1.z, s1.w);
      unpack2(acc.s2a, s2.x, s2.y);
      unpack2(acc.s2b, s2.z, s2.w);
      float l0, l1, l2, l3;
      unpack2(lacc.la, l0, l1);
      unpack2(lacc.lb, l2, l3);
      const double cons = (double)((s2.x - s1.x * s1.x * p.inv_M) + (s2.y - s1.y * s1.y * p.inv_M) +
                                   (s2.z - s1.z * s1.z * p.inv_M) + (s2.w - s1.w * s1.w * p.inv_M));
      const double loss = (double)((l0 + l1) + (l2 + l3));
      if constexpr (kReg > 0) {
#pragma unroll
        for (int kk = 0; kk < kReg; ++kk) {  // (k is known only at run time: predicated adds keep the sums in registers)
          if (kk == k) {
            acc_cons[kk] += cons;
            acc_loss[kk] += loss;
          }
        }
        return;
      }
      // lanes 0-15 go on with the one sum, lanes 16-31 with the other
      const bool low = lane < 16;
      double keep = (low ? cons : loss) + __shfl_xor_sync(0xffffffffu, low ? loss : cons, 16);
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, off);
      if ((lane & 15) == 0) s_tel[(k * nwarps + warp) * 2 + (lane >> 4)] += keep;
    };
    // (a test for padding lanes in every row would keep the rows' instructions apart: the one warp that has
    // any, or columns behind the last, runs its own instance of the round)
    if (__all_sync(0xffffffffu, lanes == 4)) {
      for (int k = 0; k + 1 < p.n_rounds; ++k) run_round(k, std::false_type(), std::false_type());
      run_round(p.n_rounds - 1, std::true_type(), std::false_type());
    } else {
      for (int k = 0; k + 1 < p.n_rounds; ++k) run_round(k, std::false_type(), std::true_type());
      run_round(p.n_rounds - 1, std::true_type(), std::true_type());
    }
    base = (base + (uint32_t)p.n_rounds) & 1u;
    fetched = have_next;
  }

  // telemetry: per round, CTA partials; the last CTA to finish sums them
#pragma unroll
  for (int k = 0; k < kReg; ++k) {
    double a = acc_cons[k], b = acc_loss[k];
    for (int off = 16; off > 0; off >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, off);
      b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if (lane == 0 && k < p.n_rounds) {
      s_tel[(k * nwarps + warp) * 2] = a;
      s_tel[(k * nwarps + warp) * 2 + 1] = b;
    }
  }
  __syncthreads();
  for (int e = tid; e < p.n_rounds * 2; e += T) {
    const int k = e >> 1;
    double a = 0.0;
    for (int w = 0; w < nwarps; ++w) a += s_tel[(k * nwarps + w) * 2 + (e & 1)];
    p.partials[((size_t)k * gridDim.x + blockIdx.x) * 2 + (e & 1)] = (e & 1) ? 0.5 * a : a;
  }
  finalize_rounds(p.partials, p.n_rounds, (double)p.inv_M, p.tel, p.slot0, p.ring, p.ticket);
}

// ------------------------------------------------------------------------- asynchronous steps
// The paper's own process (Eq. 17): at a global step ONE worker i applies Eq. 15-16 to its
// replica, in place, with the peer's current replica; every other replica is unchanged.  A
// launch carries up to kMaxStepEvents consecutive global steps that touch disjoint replicas
// (no step writes a row another step of the launch reads or writes), so their order inside
// the launch does not matter.  16 bytes of HBM traffic per element: nothing is shared.
constexpr int kMaxStepEvents = 32;

struct StepEvent {
  int32_t worker, peer;
  uint32_t iter_lo, ctr3;  // the worker's local iteration, as Philox counter words of the noise stream
  float w;                 // pull weight w_im (0 on a self-draw)
};

struct StepParams {
  float4* x;        // [M][ldq] replicas (16-byte column groups), updated in place
  const float4* c;  // [M][ldq]
  int64_t nq;
  uint32_t row_bytes;
  int32_t tail;     // d % (4 kHalves)
  float alpha, sigma;
  uint32_t q_offset;
  int32_t n_events;
  StepEvent ev[kMaxStepEvents];
  PhiloxKeys keys;
};

template <int kObjective, int kHalves>
__global__ void __launch_bounds__(256) step_kernel(const StepParams p) {
  const StepEvent& e = p.ev[blockIdx.y];
  const uint64_t row_i = (uint64_t)(uint32_t)e.worker * p.row_bytes;
  const uint64_t row_m = (uint64_t)(uint32_t)e.peer * p.row_bytes;
  char* xb = reinterpret_cast<char*>(p.x);
  const char* cb = reinterpret_cast<const char*>(p.c);
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < p.nq; q += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t off = (uint64_t)q * 16;
    const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(xb + row_i + off);
    const ulonglong2 xm = *reinterpret_cast<const ulonglong2*>(xb + row_m + off);
    ulonglong2 cv = make_ulonglong2(0ull, 0ull);
    if (kObjective == 1) cv = __ldg(reinterpret_cast<const ulonglong2*>(cb + row_i + off));
    const bool ragged = (p.tail != 0) && (q == p.nq - 1);
    ulonglong2 o;
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      pair_t ta, tb;
      const ulonglong2 noise = draw_noise<kObjective, kFunnel>(p.sigma, p.keys, e.iter_lo, e.ctr3, (uint32_t)q * kHalves + h + p.q_offset,
                                                      (uint32_t)e.worker, live_lanes(ragged, p.tail, h));
      const ulonglong2 oh = update_core<kObjective, kFunnel>(p.alpha, noise, group_half<kHalves>(xv, h), group_half<kHalves>(cv, h),
                                                    group_half<kHalves>(xm, h), e.w, ta, tb);
      if (kHalves == 1) o = oh;
      else if (h == 0) o.x = narrow_bf16x4(oh);
      else o.y = narrow_bf16x4(oh);
    }
    *reinterpret_cast<ulonglong2*>(xb + row_i + off) = o;
  }
}

// Many consecutive global steps on resident columns: given who acts and whom it pulls from, every column evolves
// on its own, so a thread that keeps one column group of ALL M rows (replicas, updated in place, and centres: 32 M
// bytes of shared memory) runs any number of steps on it without a barrier.  step_kernel moves 16 bytes per element
// and step and is bound by HBM at 27 us per step of 11.2 M elements; here a launch moves 12 M bytes per column
// element for all of its steps, and the noise (drawn a step ahead) is what takes the time.  Short vectors gain more:
// one launch for all steps instead of one for every few that touch disjoint replicas.
constexpr int kStepTileEvents = 160;  // of one launch: they travel as a kernel argument
struct StepTileParams {
  char* x;          // replicas, updated in place, row stride row_bytes
  const char* c;
  int64_t nq, n_tiles;  // column groups of four elements per row; tiles of blockDim of them
  uint32_t row_bytes;
  int32_t M, tail;  // tail = d % 4
  float alpha, sigma;
  uint32_t q_offset;
  int32_t n_events;
  PhiloxKeys keys;
  StepEvent ev[kStepTileEvents];  // (all of one high word of the iteration: the same ctr3)
};
// Noise: column and event parts of its first products are worked out once per column and once per event (noise_column,
// noise_start); 16 of 20 wide multiplies are left (8 x 11,173,962 elements, 128 steps: 1,603 us, 1,493 so).
// Dynamic shared memory: events (offset of the worker's row, of the peer's, weight, low word of the iteration's product) int4[n]
// and noise_start uint2[n], what happens to each row (1: written, 2: read), slabs float4[2][M][blockDim].
__host__ __device__ inline uint32_t step_tile_head(int events, int64_t M) { return (uint32_t)((events * 24 + M + 127) & ~(int64_t)127); }

template <int kObjective, bool kBf16>
__global__ void __launch_bounds__(256, 2) step_tiles_kernel(const __grid_constant__ StepTileParams p) {
  constexpr uint32_t kGroupBytes = kBf16 ? 8u : 16u;
  constexpr int kAhead = 4;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int tid = threadIdx.x, T = blockDim.x, M = p.M, n = p.n_events;
  const uint32_t stride = (uint32_t)T * 16u, plane = (uint32_t)M * stride;
  int4* s_ev = reinterpret_cast<int4*>(smem_raw);
  uint2* s_start = reinterpret_cast<uint2*>(s_ev + n);
  unsigned char* s_use = smem_raw + (size_t)n * 24;
  unsigned char* const x = smem_raw + step_tile_head(n, M) + (uint32_t)tid * 16u;  // this thread's column, row i at i * stride
  unsigned char* const cen = x + plane;
  for (int i = tid; i < M; i += T) s_use[i] = 0;
  for (int e = tid; e < n; e += T) {
    const StepEvent& ev = p.ev[e];
    s_ev[e] = make_int4((int)((uint32_t)ev.worker * stride), (int)((uint32_t)ev.peer * stride), __float_as_int(ev.w), (int)(kPhiloxMul1 * ev.iter_lo));
    const uint64_t start = noise_start((uint32_t)ev.worker, ev.iter_lo, p.keys);
    s_start[e] = make_uint2((uint32_t)start, (uint32_t)(start >> 32));
  }
  __syncthreads();
  for (int e = tid; e < n; e += T) s_use[p.ev[e].peer] = 2;
  __syncthreads();
  for (int e = tid; e < n; e += T) s_use[p.ev[e].worker] = 3;
  __syncthreads();

  for (int64_t tile = blockIdx.x; tile < p.n_tiles; tile += gridDim.x) {
    const int64_t q = tile * T + tid;
    if (q >= p.nq) continue;  // (threads are independent)
    char* const xq = p.x + (uint64_t)q * kGroupBytes;
    const char* const cq = p.c + (uint64_t)q * kGroupBytes;
#pragma unroll 4
    for (int i = 0; i < M; ++i) {
      const int use = s_use[i];
      const uint64_t at = (uint64_t)(uint32_t)i * p.row_bytes;
      const uint32_t to = (uint32_t)i * stride;
      if (kBf16) {
        if (use & 2) *reinterpret_cast<ulonglong2*>(x + to) = widen_bf16x4(*reinterpret_cast<const unsigned long long*>(xq + at));
        if (use & 1) *reinterpret_cast<ulonglong2*>(cen + to) = widen_bf16x4(__ldg(reinterpret_cast<const unsigned long long*>(cq + at)));
      } else {
        if (use & 2) cp_async_16_stream(x + to, xq + at);
        if (use & 1) cp_async_16_stream(cen + to, cq + at);
      }
    }
    cp_async_wait_all();
    const NoiseColumn column = noise_column((uint32_t)q + p.q_offset, p.ev[0].ctr3, p.keys);
    const int live = live_lanes((p.tail != 0) && (q == p.nq - 1), p.tail, 0);
    auto draw = [&](int e) {  // event e's noise
      ulonglong2 v = make_ulonglong2(0ull, 0ull);
      if (kObjective == 1) {
        const uint2 start = s_start[e];
        v = scaled_normals4<kFunnel>(noise_words(noise_base_of_product(column, (uint32_t)s_ev[e].w, p.keys), start.x | (uint64_t)start.y << 32, p.keys), p.sigma);
        if (live < 4) v = mask_lanes(v, live);
      }
      return v;
    };
    auto step = [&](int e, ulonglong2 noise) {
      const int4 d = s_ev[e];
      pair_t ta, tb;
      const ulonglong2 o = update_core<kObjective, kFunnel>(p.alpha, noise, *reinterpret_cast<const ulonglong2*>(x + (uint32_t)d.x),
                                                   *reinterpret_cast<const ulonglong2*>(cen + (uint32_t)d.x),
                                                   *reinterpret_cast<const ulonglong2*>(x + (uint32_t)d.y), __int_as_float(d.z), ta, tb);
      *reinterpret_cast<ulonglong2*>(x + (uint32_t)d.x) = kBf16 ? widen_bf16x4(narrow_bf16x4(o)) : o;
    };
    // The steps depend on one another, their noise does not: it is drawn kAhead events at a time, as many chains of
    // multiplies and special functions side by side (11.2 M elements: 13.3 us per step with two at a time,
    // 12.8 with four).
    int e = 0;
    for (; e + kAhead <= n; e += kAhead) {
      ulonglong2 noise[kAhead];
#pragma unroll
      for (int a = 0; a < kAhead; ++a) noise[a] = draw(e + a);
#pragma unroll
      for (int a = 0; a < kAhead; ++a) step(e + a, noise[a]);
    }
    for (; e < n; ++e) step(e, draw(e));
#pragma unroll 4
    for (int i = 0; i < M; ++i) {
      if (!(s_use[i] & 1)) continue;
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(x + (uint32_t)i * stride);
      const uint64_t at = (uint64_t)(uint32_t)i * p.row_bytes;
      if (kBf16) *reinterpret_cast<unsigned long long*>(xq + at) = narrow_bf16x4(v);
      else *reinterpret_cast<ulonglong2*>(xq + at) = v;
    }
  }
}

}  // namespace netmax
