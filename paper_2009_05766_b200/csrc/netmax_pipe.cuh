// Rounds of small problems on resident tiles, noise and telemetry beside them.
//
// Given the peer draws, every column of the M x d state evolves on its own (Eq. 16 is elementwise), so a WARP that holds
// all M rows of G column groups (four elements each) can run any number of rounds on them and meets nobody: a pull reads
// a row that another lane of the same warp wrote a round earlier (__syncwarp).  What is left of a round on that warp is
// the serial chain itself -- read the peer's value, two dependent sums, write.  The gradient noise, three quarters of a
// round's instructions, depends on no replica, and the telemetry of a round only on states that are there already: both
// are done by other warps of the CTA.
//
//   moving warps    one tile each; in registers the tile's own rows and centres, in shared memory a ring of states
//   helping warps   while batch b of rounds runs: the noise and draws of batch b + 1, the telemetry of batch b - 1
//
// All warps meet (meet_at_batch) once per batch of rounds, not once per round.
//
// Bound by latency: a round takes the moving warp about 125 cycles with one row per lane (the peer's value by a shuffle,
// the noise and draws of the next round read under it), a batch about 670 besides.  4 x 4,096 elements, 500 rounds: 281 us
// with the rows of a tile spread over warps that meet every round (tile_rounds_kernel, 1,106 cycles per round, most of it
// one warp's chain of noise and then sums), 49 us here.  Above some ten rows of 32 column groups per SM the instructions
// of the helping warps are what takes the time (95 cycles per such row and SM), and tile_rounds_kernel needs fewer.
#pragma once
#include "netmax_tiles.cuh"

namespace netmax {

struct PipeParams {
  const char* x_cur;      // replicas at the start of the first round, row stride row_bytes
  char* x_nxt;            // replicas after the last round
  char* mirror;           // copy of them in page-locked host memory (fp32 state); may be NULL
  const char* c;
  const int2* draws;      // ring of (peer, bits of the pull weight), [ring][M]
  double* partials;       // [n_rounds][gridDim.x][2]: telemetry shares of every CTA
  int64_t slot0, ring;
  uint64_t first_round;
  int32_t n_rounds;
  int32_t n_tiles;        // tiles of G column groups of four elements, at most gridDim.x x movers: mover w has tile blockIdx.x + w gridDim.x
  int64_t nq;
  uint32_t row_bytes;
  int32_t M, tail;        // tail = d % 4
  int32_t G, log2G;       // column groups per tile (a power of two, at most 32)
  int32_t movers, batch;  // moving warps of a CTA, rounds per batch
  float alpha, sigma, inv_M;  // sigma: the noise scale sigma sqrt(2 ln 2)
  uint32_t q_offset;
  PhiloxKeys keys;
};

constexpr int kPipeThreads = 512;
constexpr int kPipeMaxRows = 8;
// The telemetry of a round: so many rows of a column are added up in fp32 at a time, then four such sums, then those.  One chain over all
// rows lost precision with their number.  Root mean square error of the consensus distance against 64-bit sums, so / one chain / the shares
// of tile_rounds_kernel: 16 x 2,048 elements 4.3e-9 / 8.1e-9 / 9.7e-9, 64 x 2,048 3.5e-9 / 1.1e-8 / 5.2e-9, 100 x 1,310 6.4e-9 / 1.8e-8 /
// 8.2e-9, 100 x 400 in bfloat16 2.6e-8 / 3.7e-7 / 2.7e-8 (one column of 100 workers: the loss 6.0e-8 / 1.6e-7 / 4.3e-8).  It costs nothing
// up to eight rows and is as fast beyond, 200 rounds of 64 x 400 elements 60.3 us / 62.3, 99 x 1,401 150.4 / 146.8; sums that go on in
// double from eight rows on took 72 and 184, from 32 on 63 and 160.
constexpr int kPipeSumRows = 8;

// Dynamic shared memory: per moving warp a ring of 2 batch + 1 states, the noise of 2 batch rounds and the centres,
// float4[rows][G] each, rows filled up to what 32 lanes of `per_lane` rows hold (what stands there is never looked at);
// draws (peer, weight) int2[2][batch][rows]; shares double[2][batch][movers][2].
__host__ __device__ inline size_t pipe_smem(int G, int per_lane, int movers, int batch) {
  return (size_t)movers * per_lane * 512 * (4 * batch + 2) + (size_t)2 * batch * (32 / G * per_lane) * 8 + (size_t)2 * batch * movers * 16;
}

// The warps of a CTA meet from two places of the program, the moving ones' loop and the helping ones': a barrier by name and number of
// threads, which says so (__syncthreads is only defined where the whole CTA takes the same branch).
__device__ __forceinline__ void meet_at_batch() { asm volatile("barrier.sync 1, %0;" ::"r"(blockDim.x) : "memory"); }

// kRows: rows per lane, ceil(M G / 32).
template <int kObjective, bool kBf16, int kRows>
__global__ void __launch_bounds__(kPipeThreads, 1) pipe_rounds_kernel(const __grid_constant__ PipeParams p) {
  constexpr uint32_t kGroupBytes = kBf16 ? 8u : 16u;  // four elements in global memory
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);  // (the same in all lanes, for the compiler too)
  const int M = p.M, G = p.G, B = p.batch, NC = p.movers, NH = warps - NC, R = 2 * B + 1, n = p.n_rounds;
  const int g = lane & (G - 1), r = lane >> p.log2G, RL = 32 >> p.log2G;
  const int rows_up = RL * kRows;            // M filled up
  constexpr uint32_t state = 512u * kRows;   // bytes of one state of a tile
  const uint32_t per_mover = state * (uint32_t)(4 * B + 2);
  int2* const s_pw = reinterpret_cast<int2*>(smem_raw + (size_t)NC * per_mover);
  double* const s_part = reinterpret_cast<double*>(s_pw + 2 * B * rows_up);
  const uint32_t lane_at = ((uint32_t)r * (uint32_t)G + (uint32_t)g) * 16u;  // this lane's first row in a state
  constexpr uint32_t step = 512u;                                            // bytes to its next one, RL rows on
  const int batches = (n + B - 1) / B;
  auto rows = [&](auto body) {
#pragma unroll
    for (int j = 0; j < kRows; ++j) body(j);
  };
  if (warp < NC) {
    unsigned char* const mine = smem_raw + (size_t)warp * per_mover;
    unsigned char* const s_noise = mine + (size_t)R * state;
    unsigned char* const s_c = s_noise + (size_t)2 * B * state;
    const int tile = (int)blockIdx.x + warp * (int)gridDim.x;
    const int64_t q = (int64_t)tile * G + g;
    const bool live = tile < p.n_tiles && q < p.nq;
    ulonglong2 x[kRows], cv[kRows];
    const uint64_t row0 = (uint64_t)(uint32_t)r * p.row_bytes, row_step = (uint64_t)(uint32_t)RL * p.row_bytes;
    if (tile < p.n_tiles) {
      rows([&](int j) {
        x[j] = cv[j] = make_ulonglong2(0ull, 0ull);
        if (live && r + j * RL < M) {
          const char* xq = p.x_cur + (uint64_t)q * kGroupBytes + row0 + j * row_step;
          const char* cq = p.c + (uint64_t)q * kGroupBytes + row0 + j * row_step;
          if (kBf16) {
            x[j] = widen_bf16x4(__ldg(reinterpret_cast<const unsigned long long*>(xq)));
            cv[j] = widen_bf16x4(__ldg(reinterpret_cast<const unsigned long long*>(cq)));
          } else {
            x[j] = __ldg(reinterpret_cast<const ulonglong2*>(xq));
            cv[j] = __ldg(reinterpret_cast<const ulonglong2*>(cq));
          }
        }
        *reinterpret_cast<ulonglong2*>(mine + lane_at + j * step) = x[j];
        *reinterpret_cast<ulonglong2*>(s_c + lane_at + j * step) = cv[j];
      });
    }
    unsigned char *cur = mine + (uint32_t)g * 16u, *const last = cur + (size_t)(R - 1) * state;  // the present state, this lane's group
    const uint32_t row_at = lane_at - (uint32_t)g * 16u;
    for (int ph = 0; ph < batches + 3; ++ph) {
      meet_at_batch();  // the noise and draws of batch ph are there
      if (ph >= batches || tile >= p.n_tiles) continue;
      const int len = min(B, n - ph * B);
      const unsigned char* nz = s_noise + (size_t)(ph & 1) * B * state + lane_at;
      const int2* pw = s_pw + (size_t)(ph & 1) * B * rows_up + r;  // (peer, weight)
      // a round's noise and draws, fetched a round ahead
      struct Ahead {
        ulonglong2 noise[kRows];
        int2 d[kRows];
      };
      auto fetch = [&](Ahead& a) {
        rows([&](int j) {
          a.noise[j] = kObjective == 1 ? *reinterpret_cast<const ulonglong2*>(nz + j * step) : make_ulonglong2(0ull, 0ull);
          a.d[j] = pw[j * RL];
        });
        nz += state;
        pw += rows_up;
      };
      auto round = [&](const Ahead& a, Ahead& next, bool more) {
        ulonglong2 xm[kRows];
        if constexpr (kRows == 1) {  // the peer's value from its lane
          const int from = (a.d[0].x << p.log2G) + g;
          xm[0].x = __shfl_sync(0xffffffffu, x[0].x, from);
          xm[0].y = __shfl_sync(0xffffffffu, x[0].y, from);
        } else {
          __syncwarp();  // the state is complete
          rows([&](int j) { xm[j] = *reinterpret_cast<const ulonglong2*>(cur + ((uint32_t)a.d[j].x << (p.log2G + 4))); });
        }
        cur = cur == last ? mine + (uint32_t)g * 16u : cur + state;
        if (more) fetch(next);
        rows([&](int j) {
          pair_t ta, tb;
          ulonglong2 o = update_core<kObjective, kFunnel>(p.alpha, a.noise[j], x[j], cv[j], xm[j], __int_as_float(a.d[j].y), ta, tb);
          if (kBf16) o = widen_bf16x4(narrow_bf16x4(o));
          x[j] = o;
          *reinterpret_cast<ulonglong2*>(cur + row_at + j * step) = o;
        });
      };
      Ahead a0, a1;
      fetch(a0);
      int k = 0;
      for (; k + 1 < len; k += 2) {
        round(a0, a1, true);
        round(a1, a0, k + 2 < len);
      }
      if (k < len) round(a0, a1, false);
    }
    if (live) {
      char* oq = p.x_nxt + (uint64_t)q * kGroupBytes + row0;
      char* mq = !kBf16 && p.mirror ? p.mirror + (uint64_t)q * kGroupBytes + row0 : nullptr;
      rows([&](int j) {
        if (r + j * RL >= M) return;
        if (kBf16) *reinterpret_cast<unsigned long long*>(oq + j * row_step) = narrow_bf16x4(x[j]);
        else *reinterpret_cast<ulonglong2*>(oq + j * row_step) = x[j];
        if (!kBf16 && mq) *reinterpret_cast<ulonglong2*>(mq + j * row_step) = x[j];
      });
    }
  } else {
    // Helping warps h = w, w + NC, ... serve mover w: everything that depends on the tile alone is worked out once.
    const int h = warp - NC, w = h % NC, first_kk = h / NC, per_tile = NH / NC;
    const int tile = (int)blockIdx.x + w * (int)gridDim.x;
    const bool busy = tile < p.n_tiles;
    const int64_t q = (int64_t)tile * G + g;
    const int live = busy && q < p.nq ? live_lanes(p.tail != 0 && q == p.nq - 1, p.tail, 0) : 0;
    const bool ragged = !__all_sync(0xffffffffu, live == 4);
    unsigned char* const tile_at = smem_raw + (size_t)w * per_mover;
    const NoiseColumn column = noise_column((uint32_t)q + p.q_offset, philox_ctr3(kTagNoise, p.first_round), p.keys);
    // the noise of kAtOnce rounds of batch ph, per_tile apart
    auto draw_noise = [&](int ph, int kk, auto at_once) {
      constexpr int kAtOnce = decltype(at_once)::value;
      NoiseBase nb[kAtOnce];
#pragma unroll
      for (int a = 0; a < kAtOnce; ++a)
        nb[a] = noise_base(column, (uint32_t)p.first_round + (uint32_t)(ph * B + kk + a * per_tile), p.keys);
      unsigned char* to = tile_at + (size_t)(R + (ph & 1) * B + kk) * state + lane_at;
      rows([&](int j) {
#pragma unroll
        for (int a = 0; a < kAtOnce; ++a) {
          ulonglong2 z = scaled_normals4<kFunnel>(noise_words(nb[a], (uint32_t)(r + j * RL), p.keys), p.sigma);
          if (ragged) z = mask_lanes(z, live);
          *reinterpret_cast<ulonglong2*>(to + (size_t)a * per_tile * state + j * step) = z;
        }
      });
    };
    constexpr int kPair = kRows <= 2 ? 2 : 1;  // (a lane's rows are independent chains, too)
    int64_t draw_slot = p.slot0 % p.ring;      // ring slot of the batch's first round
    int tel_slot = 0;                          // ring slot of the first state of the batch whose telemetry is next
    for (int ph = 0; ph < batches + 3; ++ph) {
      const int len = min(B, n - ph * B);
      auto fetch_draws = [&]() {
        for (int kk = h; kk < len; kk += NH) {
          const int64_t slot = draw_slot + kk >= p.ring ? draw_slot + kk - p.ring : draw_slot + kk;
          for (int i = lane; i < rows_up; i += 32) {
            int2* to = s_pw + ((ph & 1) * B + kk) * rows_up + i;
            if (i < M) cp_async_8(to, p.draws + slot * M + i);
            else *to = make_int2(0, 0);
          }
        }
        draw_slot = draw_slot + len >= p.ring ? draw_slot + len - p.ring : draw_slot + len;
      };
      if (ph > 0 && ph < batches) fetch_draws();
      if (kObjective == 1 && busy) {
        for (int kk = first_kk; kk < len; kk += kPair * per_tile) {
          if (kPair == 2 && kk + per_tile < len) draw_noise(ph, kk, std::integral_constant<int, 2>());
          else draw_noise(ph, kk, std::integral_constant<int, 1>());
        }
      }
      if (ph == 0) {
        wait_for_previous();  // (the noise of the first batch beside the sampler)
        fetch_draws();
      }
      if (ph >= 2 && ph < batches + 2) {  // telemetry of batch ph - 2, whose last state is there: a lane adds up a column group
        const int rounds = min(B, n - (ph - 2) * B);
        for (int k0 = first_kk << (5 - p.log2G); k0 < rounds; k0 += per_tile << (5 - p.log2G)) {
          const int kk = k0 + r;
          double s2 = 0.0, loss = 0.0;
          if (kk < rounds && busy) {
            const unsigned char* xs = tile_at + (size_t)(tel_slot + kk >= R ? tel_slot + kk - R : tel_slot + kk) * state + (uint32_t)g * 16u;
            const unsigned char* cs = tile_at + (size_t)(R + 2 * B) * state + (uint32_t)g * 16u;
            const ulonglong2 pivot = *reinterpret_cast<const ulonglong2*>(xs);  // row 0
            ColAcc acc;
            LossAcc lacc;
            auto add_row = [&](ColAcc& to, LossAcc& lto) {
              const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(xs);
              const ulonglong2 c4 = *reinterpret_cast<const ulonglong2*>(cs);
              row_update<2, 0>(0.f, pivot, xv, c4, xv, pivot, 0.f, to, lto);
              xs += (uint32_t)G * 16u;
              cs += (uint32_t)G * 16u;
            };
            auto add = [](ColAcc& to, LossAcc& lto, const ColAcc& from, const LossAcc& lfrom) {
              to.s1a = add2(to.s1a, from.s1a);
              to.s1b = add2(to.s1b, from.s1b);
              to.s2a = add2(to.s2a, from.s2a);
              to.s2b = add2(to.s2b, from.s2b);
              lto.la = add2(lto.la, lfrom.la);
              lto.lb = add2(lto.lb, lfrom.lb);
            };
            if (M <= kPipeSumRows) {
#pragma unroll 4
              for (int i = 0; i < M; ++i) add_row(acc, lacc);
            } else for (int left = M; left > 0;) {  // (what is short of a whole group or part comes first)
              const int group = (left - 1) % (4 * kPipeSumRows) + 1, odd = group % kPipeSumRows;
              ColAcc of_group;
              LossAcc lof_group;
#pragma unroll 4
              for (int k = 0; k < odd; ++k) add_row(of_group, lof_group);
              for (int k = odd; k < group; k += kPipeSumRows) {
                ColAcc part;
                LossAcc lpart;
#pragma unroll
                for (int e = 0; e < kPipeSumRows; ++e) add_row(part, lpart);
                add(of_group, lof_group, part, lpart);
              }
              add(acc, lacc, of_group, lof_group);
              left -= group;
            }
            float4 s1, q2;
            float l0, l1, l2, l3;
            unpack2(acc.s1a, s1.x, s1.y);
            unpack2(acc.s1b, s1.z, s1.w);
            unpack2(acc.s2a, q2.x, q2.y);
            unpack2(acc.s2b, q2.z, q2.w);
            unpack2(lacc.la, l0, l1);
            unpack2(lacc.lb, l2, l3);
            // sum_i (x_i - xbar)^2 = sum_i (x_i - a)^2 - (sum_i (x_i - a))^2 / M per column
            s2 = (double)((fmaf(-s1.x * p.inv_M, s1.x, q2.x) + fmaf(-s1.y * p.inv_M, s1.y, q2.y)) +
                          (fmaf(-s1.z * p.inv_M, s1.z, q2.z) + fmaf(-s1.w * p.inv_M, s1.w, q2.w)));
            loss = (double)((l0 + l1) + (l2 + l3));
          }
          for (int off = G >> 1; off > 0; off >>= 1) {
            s2 += __shfl_xor_sync(0xffffffffu, s2, off);
            loss += __shfl_xor_sync(0xffffffffu, loss, off);
          }
          if (g == 0 && kk < rounds) {
            double* out = s_part + (((ph & 1) * B + kk) * NC + w) * 2;
            out[0] = s2;
            out[1] = 0.5 * loss;
          }
        }
        tel_slot = tel_slot + B >= R ? tel_slot + B - R : tel_slot + B;
      }
      if (ph >= 3) {  // the tiles' shares of the rounds of batch ph - 3, in order
        const int b = ph - 3, rounds = min(B, n - b * B);
        for (int e = h * 32 + lane; e < rounds * 2; e += NH * 32) {
          const double* in = s_part + (((ph - 1) & 1) * B + (e >> 1)) * NC * 2 + (e & 1);
          double a = 0.0;
          for (int w = 0; w < NC; ++w) a += in[2 * w];
          double* out = p.partials + ((size_t)(b * B + (e >> 1)) * gridDim.x + blockIdx.x) * 2 + (e & 1);
          *out = a;
        }
      }
      cp_async_wait_all();
      meet_at_batch();
    }
  }
}

}  // namespace netmax
