// Rounds on resident tiles whose rows are shared out over the threads of a CTA (any number of workers
// that fits on chip: 48 bytes per worker and column group).
//
// Given the peer draws, every column of the M x d state evolves on its own (Eq. 16 is elementwise), so a
// CTA that holds ALL M rows of G column groups (four elements each) in shared memory can run any number
// of rounds on them.  Thread (g, r) owns the rows r, r + RL, ... of group g; a pull reads the peer's row of
// the same group, which another thread wrote a round earlier, so rounds are separated by a barrier.
//
// What bounds it, and why it is laid out this way.  Three quarters of a round's instructions draw the
// gradient noise, which depends on no replica: a thread draws the noise of its rows for the NEXT round
// between arriving at the round's barrier and waiting for it (an mbarrier, so that the two are apart), and
// carries it over in registers (4 per row; at most kRows rows per thread).  The barrier, the slowest warp
// and the telemetry sums then hide behind work that has to be done anyway.  On 64 x 11.2 M elements the
// same tile with noise drawn inside the round and a CTA barrier measured 1,685 us per round, rows over a
// cluster of eight CTAs 1,380.  What of the noise's first products depends on the column alone is worked out once per tile, and a
// thread's rows lie a constant distance apart: per row of a column group and scheduler 214 -> 207 cycles with 64 workers (bfloat16
// state 224 -> 216), 93 in bfloat16 247 -> 236, 1,000 workers 205 -> 196, 4,096 200 -> 193.
#pragma once
#include "netmax_kernels.cuh"

namespace netmax {

// ---- mbarrier ----------------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("{\n.reg .b64 t;\nmbarrier.arrive.shared::cta.b64 t, [%0];\n}" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
               : "=r"(ok)
               : "r"(bar), "r"(parity)
               : "memory");
  return ok != 0;
}
// Every warp of the CTA arrives unconditionally, so the wait ends; it is bounded all the same, and one that
// runs out is reported (the replicas are then not valid).
constexpr uint32_t kTileSpinLimit = 1u << 22;
__device__ __forceinline__ void mbar_wait(uint32_t bar, uint32_t parity, unsigned int* error) {
  for (uint32_t it = 0; it < kTileSpinLimit; ++it)
    if (mbar_try_wait(bar, parity)) return;
  *reinterpret_cast<volatile unsigned int*>(error) = 1u;
}

struct TileParams {
  const char* x_cur;      // replicas at the start of the first round, row stride row_bytes
  char* x_nxt;            // replicas after the last round
  char* mirror;           // copy of them in page-locked host memory (fp32 state); may be NULL
  const char* c;
  const int2* draws;      // ring of (peer, bits of the pull weight), [ring][M]
  double* partials;       // [n_rounds][gridDim.x][2]: telemetry shares of every CTA
  double* tel;            // telemetry ring; written by the last CTA when finalize is set
  unsigned int* ticket;   // last-CTA-done counter (0 between launches)
  unsigned int* error;
  int64_t slot0, ring;
  uint64_t first_round;   // (its high word is that of all rounds of the launch)
  int32_t n_rounds;
  int64_t nq, n_tiles;    // column groups of four elements per row; tiles of G of them
  uint32_t row_bytes;
  int32_t M, tail;        // tail = d % 4
  int32_t G, log2G;       // column groups per tile (a power of two, at most 32)
  int32_t pre_reduce;     // sums are added over the lanes of a warp first (scratch for G entries per warp, not 32)
  int32_t finalize;
  int64_t units;          // > 0: tiles are cut, every CTA runs this many rounds of tiles (see Piece)
  unsigned int* cut;      // [gridDim.x]: raised by a CTA that has run its share of a cut tile (0 before the launch)
  float alpha, sigma, inv_M;   // sigma: the noise scale sigma sqrt(2 ln 2)
  uint32_t q_offset;
  PhiloxKeys keys;
};

// What a CTA runs: rounds [k0, k1) of a tile.  With many tiles a CTA takes every gridDim.x-th one, all rounds.
// With few of them (units > 0) that leaves some CTAs a whole tile more than others -- 256 tiles on 148 CTAs
// take as long as 296 -- so tiles are cut: laid end to end, tile by tile and round by round, the work is dealt
// out in equal lengths, each at least one tile's.  A cut tile's first rounds are the END of CTA b - 1's length
// and its last rounds the BEGINNING of CTA b's; every CTA runs its length from the far end, so that b - 1
// starts with its share and b finishes with the rest, long after the share is there.  The state between them
// goes through x_nxt; b waits (bounded) for a flag of b - 1, which by then waits for nobody, and the launch is
// cooperative, so that both are resident.  4096 x 1024 elements: 8.7 -> 7.5 us per round.
struct Piece {
  int64_t tile;
  int32_t k0, k1;
};
// The n-th piece of this CTA; false: there is none.
__device__ __forceinline__ bool tile_piece(const TileParams& p, int n, Piece& out) {
  const int64_t b = blockIdx.x, R = p.n_rounds;
  out.k0 = 0;
  out.k1 = p.n_rounds;
  if (p.units == 0) {
    out.tile = b + (int64_t)n * gridDim.x;
    return out.tile < p.n_tiles;
  }
  const int64_t all = p.n_tiles * R;
  const int64_t lo = min(all, b * p.units), hi = min(all, lo + p.units);
  const int32_t k_lo = (int32_t)(lo % R), k_hi = (int32_t)(hi % R);
  const int64_t first = (lo + R - 1) / R, last = hi / R;  // whole tiles [first, last)
  if (k_hi > 0) {  // the share of tile `last` (a length is at least one tile's, so it begins in this one)
    if (n == 0) {
      out.tile = last;
      out.k1 = k_hi;
      return true;
    }
    --n;
  }
  if (n < last - first) {
    out.tile = first + n;
    return true;
  }
  if (n == last - first && k_lo > 0) {  // the rest of the tile that CTA b - 1 begins
    out.tile = first - 1;
    out.k0 = k_lo;
    return true;
  }
  return false;
}

// Threads a CTA of the instance with `rows` rows per thread may have (and an SM holds): the registers of a row
// decide.
__host__ __device__ constexpr int tile_max_threads(int rows) { return rows <= 8 ? 512 : rows <= 10 ? 448 : 384; }
constexpr int kTileMaxRows = 16;
__host__ __device__ constexpr int log2_of(int g) { return g <= 1 ? 0 : 1 + log2_of(g >> 1); }
// What the shares of a round are added up in: fp32 sums are a thread's own, and those of column sums.  Double with five
// rows per thread and more (long vectors of fp32 state up to 88 workers, whose sums across threads have always been
// double, run on nothing else; an error of 1.2e-9 in the loss of 64 x 262,147 elements is 6e-11 with it).  With fewer
// rows (short vectors) it would cost 8 %, and with eleven, where the compiler's schedule falls apart, 18 % (4096 x 1024
// elements: 6.5 us per round, 7.7).  Four loads of a lane are in flight (4096 x 1024: 7.04 us per round without, 5.87;
// eight: 7.13).
constexpr int kShareUnroll = 4;
__host__ __device__ constexpr bool tile_wide(int rows) { return rows > 4 && rows != 11; }
// Few rows per thread make a round short, and what is not the round itself counts: draws are fetched two rounds
// ahead, and the sums of a round are added after the NEXT round's arrival, beside its noise, which takes a third
// buffer (32 x 1000 elements: 0.79 -> 0.68 us per round).  With more rows the buffer is better kept for slabs.
__host__ __device__ constexpr bool tile_far(int rows) { return rows <= 4; }

// Dynamic shared memory: slabs float4[3][M][G] (replicas of even and of odd rounds, centres), then two or three
// buffers of telemetry shares, each float4[E] + float2[E] with E = warps x (pre_reduce ? G : 32).
__host__ __device__ inline uint32_t tile_share_entries(int threads, int G, bool pre_reduce) {
  return (uint32_t)(threads >> 5) * (uint32_t)(pre_reduce ? G : 32);
}
__host__ __device__ inline size_t tile_smem(int64_t M, int threads, int G, bool pre_reduce, int rows) {
  return (size_t)48 * M * G + (size_t)(tile_far(rows) ? 72 : 48) * tile_share_entries(threads, G, pre_reduce);
}

// kRows: rows per thread, ceil(M / RL).  Exact, so that only a thread's LAST row can be missing: rows before it
// run without a test between them and the scheduler can mix their instructions (with a test per row the same
// rows took 282 cycles each instead of 195).
// kG, kWarps: column groups per tile and warps per CTA where the instance is made for one shape (0: any).  A thread's addresses are
// then one register and constants: per row of a column group and scheduler, any shape / its own, 40 workers (32 groups, 4 warps)
// 214 / 195 cycles, 54 (32, 8) 221 / 208, 64 (32, 8) 207 / 201 (bfloat16 state 216 / 212), 150 (8, 4) 223 / 203, 300 (4, 4) 225 /
// 208.  Shapes that were measured to gain 3 % and more have such instances (tile_shape_of_its_own): four warps of ten rows, which the plan
// chooses more often than any other, and eight of seven and eight (50 to 64 workers where few tiles fall on a CTA).  Twelve warps gained
// 0 to 2 %, six rows per thread lost 2 %; four warps of nine and of twelve rows were not measured.  The instances of ten rows spill (12 to 88
// bytes per thread in fp32, 124 to 144 in bfloat16; any shape's 24 and 84) and gain all the same.
__host__ __device__ constexpr bool tile_shape_of_its_own(int rows, int G, int warps) {
  return (warps == 4 && rows == 10) || (warps == 8 && G == 32 && (rows == 7 || rows == 8));
}
template <int kObjective, bool kBf16, int kRows, int kG = 0, int kWarps = 0>
__global__ void __launch_bounds__(tile_max_threads(kRows), 1) tile_rounds_kernel(const TileParams p) {
  constexpr uint32_t kGroupBytes = kBf16 ? 8u : 16u;  // four elements in global memory
  constexpr bool kFar = tile_far(kRows);
  constexpr uint32_t kBuffers = kFar ? 3u : 2u;
  using Sum = typename std::conditional<tile_wide(kRows), double, float>::type;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long s_bar;
  const int tid = threadIdx.x, T = kWarps ? kWarps * 32 : blockDim.x, M = p.M, G = kG ? kG : p.G;
  const int log2G = kG ? log2_of(kG) : p.log2G;
  const int lane = tid & 31, warp = tid >> 5, nwarps = T >> 5;
  const int g = tid & (G - 1), r = tid >> log2G, RL = T >> log2G;
  const uint32_t stride = (uint32_t)G * 16u;    // bytes between consecutive rows of a slab
  const uint32_t plane = (uint32_t)M * stride;
  const uint32_t step = (uint32_t)T * 16u;      // bytes between consecutive rows of a thread: RL rows on
  const bool full = r + (kRows - 1) * RL < M;   // has this thread a last row?
  const uint64_t row_step = (uint64_t)(uint32_t)RL * p.row_bytes, row_first = (uint64_t)(uint32_t)r * p.row_bytes;
  unsigned char* const col = smem_raw + (uint32_t)g * 16u;
  unsigned char* const own = smem_raw + (uint32_t)tid * 16u;  // row r of group g
  const uint32_t E = tile_share_entries(T, G, p.pre_reduce != 0);
  float4* const s_sum = reinterpret_cast<float4*>(smem_raw + 3u * plane);     // [kBuffers][E]
  float2* const s_two = reinterpret_cast<float2*>(s_sum + kBuffers * E);      // [kBuffers][E]
  const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&s_bar);
  if (tid == 0) mbar_init(bar, (uint32_t)nwarps);
  wait_for_previous();
  __syncthreads();

  int2 draw[kRows], draw_far[kFar ? kRows : 1];
  ulonglong2 noise[kRows];

  // body(j) for the rows of this thread
  auto rows = [&](auto body) {
#pragma unroll
    for (int j = 0; j < kRows - 1; ++j) body(j);
    if (full) body(kRows - 1);
  };
  int64_t slot = 0;  // ring slot of the draws to be loaded next
  auto load_draws = [&](int2* into) {
    const int2* src = p.draws + slot * M + r;
    rows([&](int j) { into[j] = __ldg(src + j * RL); });
    slot = slot + 1 == p.ring ? 0 : slot + 1;
  };
  auto first_draws = [&](int k) {  // of a piece that starts at round k
    slot = (p.slot0 + k) % p.ring;
    load_draws(draw);
    if (kFar) load_draws(draw_far);
  };
  auto next_draws = [&]() {  // (past the last round what comes is not used)
    if (kFar) {
      rows([&](int j) { draw[j] = draw_far[j]; });
      load_draws(draw_far);
    } else {
      load_draws(draw);
    }
  };
  // (scalar steps and the funnel shift: without it 4096 x 1024 elements take 19 % longer)
  NoiseColumn column;  // of the group whose noise is drawn
  auto enter_column = [&](int64_t q) { column = noise_column((uint32_t)q + p.q_offset, philox_ctr3(kTagNoise, p.first_round), p.keys); };
  auto next_noise = [&](int64_t q, int k) {
    if (kObjective != 1) return;
    const NoiseBase nb = noise_base(column, (uint32_t)(p.first_round + (uint64_t)k), p.keys);
    rows([&](int j) { noise[j] = scaled_normals4<kFunnel>(noise_words(nb, (uint32_t)(r + j * RL), p.keys), p.sigma); });
    if (p.tail != 0 && q == p.nq - 1)
      rows([&](int j) { noise[j] = mask_lanes(noise[j], p.tail); });
  };
  // telemetry of one round: this warp adds the shares of all threads (lane -> entries lane, lane + 32, ...,
  // which belong to column group lane % G) and leaves the CTA's two sums
  auto add_shares = [&](uint32_t buf, int k) {
    float4 s1 = make_float4(0.f, 0.f, 0.f, 0.f);
    Sum s2 = 0, loss = 0;
    auto add = [&](uint32_t e) {
      const float4 a = s_sum[buf * E + e];
      const float2 b = s_two[buf * E + e];
      s1.x += a.x; s1.y += a.y; s1.z += a.z; s1.w += a.w;
      s2 += (Sum)b.x;
      loss += (Sum)b.y;
    };
    if (kRows < 12) {
#pragma unroll kShareUnroll
      for (uint32_t e = lane; e < E; e += 32) add(e);
    } else {  // (the compiler's choice: 8 % faster than four with 93 x 721,603 elements)
      for (uint32_t e = lane; e < E; e += 32) add(e);
    }
    for (int off = 16; off >= G; off >>= 1) {
      s1.x += __shfl_xor_sync(0xffffffffu, s1.x, off);
      s1.y += __shfl_xor_sync(0xffffffffu, s1.y, off);
      s1.z += __shfl_xor_sync(0xffffffffu, s1.z, off);
      s1.w += __shfl_xor_sync(0xffffffffu, s1.w, off);
    }
    // sum_i (x_i - xbar)^2 = sum_i (x_i - a)^2 - (sum_i (x_i - a))^2 / M per column
    if (lane < G) s2 -= (Sum)(s1.x * s1.x + s1.y * s1.y + s1.z * s1.z + s1.w * s1.w) * (Sum)p.inv_M;
    double* out = p.partials + ((size_t)k * gridDim.x + blockIdx.x) * 2;
    if constexpr (tile_wide(kRows)) {  // lanes 0-15 go on with the one sum, lanes 16-31 with the other
      const bool low = lane < 16;
      Sum keep = (low ? s2 : loss) + __shfl_xor_sync(0xffffffffu, low ? loss : s2, 16);
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, off);
      if ((lane & 15) == 0) asm volatile("red.global.add.f64 [%0], %1;" ::"l"(out + (lane >> 4)), "d"(low ? (double)keep : 0.5 * (double)keep) : "memory");
    } else {
      for (int off = 16; off > 0; off >>= 1) {
        s2 += __shfl_down_sync(0xffffffffu, s2, off);
        loss += __shfl_down_sync(0xffffffffu, loss, off);
      }
      if (lane == 0) {
        asm volatile("red.global.add.f64 [%0], %1;" ::"l"(out), "d"((double)s2) : "memory");
        asm volatile("red.global.add.f64 [%0], %1;" ::"l"(out + 1), "d"(0.5 * (double)loss) : "memory");
      }
    }
  };
  for (int k = tid; k < p.n_rounds; k += T)
    reinterpret_cast<double2*>(p.partials)[(size_t)k * gridDim.x + blockIdx.x] = make_double2(0.0, 0.0);
  __syncthreads();

  // a piece's rows into slab `base` (once CTA b - 1 has done its share of a cut tile), the draws and the noise of
  // its first round; then arrives
  auto load_piece = [&](const Piece& pc, uint32_t base) {
    if (pc.k0 > 0) {
      if (tid == 0) {
        uint32_t it = 0;
        while (*reinterpret_cast<volatile unsigned int*>(p.cut + blockIdx.x - 1) == 0u && ++it < kTileSpinLimit) __nanosleep(64);
        if (it == kTileSpinLimit) *reinterpret_cast<volatile unsigned int*>(p.error) = 1u;
        __threadfence();
      }
      __syncthreads();
    }
    const int64_t q = pc.tile * G + g;
    if (q < p.nq) {
      const char* xq = (pc.k0 == 0 ? p.x_cur : p.x_nxt) + (uint64_t)q * kGroupBytes + row_first;
      const char* cq = p.c + (uint64_t)q * kGroupBytes + row_first;
      rows([&](int j) {
        unsigned char* sx = own + base * plane + (uint32_t)j * step;
        unsigned char* sc = own + 2u * plane + (uint32_t)j * step;
        if (kBf16) {
          *reinterpret_cast<ulonglong2*>(sx) = widen_bf16x4(__ldcg(reinterpret_cast<const unsigned long long*>(xq + j * row_step)));
          *reinterpret_cast<ulonglong2*>(sc) = widen_bf16x4(__ldg(reinterpret_cast<const unsigned long long*>(cq + j * row_step)));
        } else {
          cp_async_16_stream(sx, xq + j * row_step);
          cp_async_16_stream(sc, cq + j * row_step);
        }
      });
    }
    first_draws(pc.k0);
    enter_column(q);
    next_noise(q, pc.k0);
    cp_async_wait_all();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
  };

  uint32_t base = 0, phase = 0, buf = 0;
  // the last round whose shares have not been added, and the warp -- a different one every round -- that does it
  int turn = 0, last_k = -1;
  Piece pc = {0, 0, 0}, next = {0, 0, 0};
  bool more = tile_piece(p, 0, pc);
  if (more) load_piece(pc, 0);
  for (int n = 1; more; ++n) {
    const int64_t q = pc.tile * G + g;
    const bool live = q < p.nq;
    more = tile_piece(p, n, next);
    const bool ahead = more && next.k0 == 0;  // the next piece's rows are fetched under this one's last round
    const int64_t q_next = next.tile * G + g;
    const bool have_next = ahead && q_next < p.nq;

    auto run_round = [&](int k, auto last_tag) {
      constexpr bool kLast = decltype(last_tag)::value;
      mbar_wait(bar, phase, p.error);  // all rows of the previous round are written
      phase ^= 1u;
      if (!kFar && last_k >= 0 && warp == turn) add_shares(buf ^ 1u, last_k);
      const uint32_t cur_off = ((base + (uint32_t)(k - pc.k0)) & 1u) * plane, nxt_off = plane - cur_off;
      ColAcc acc;
      LossAcc lacc;
      if (kLast && have_next) {  // the next tile's replicas into the slab this round does not write
        const char* xq = p.x_cur + (uint64_t)q_next * kGroupBytes + row_first;
        rows([&](int j) {
          unsigned char* sx = own + nxt_off + (uint32_t)j * step;
          if (kBf16) cp_async_8(sx, xq + j * row_step);
          else cp_async_16_stream(sx, xq + j * row_step);
        });
      }
      if (live) {
        const unsigned char* cur = col + cur_off;
        const ulonglong2 pivot = *reinterpret_cast<const ulonglong2*>(cur);  // row 0
        char* oq = p.x_nxt + (uint64_t)q * kGroupBytes + row_first;
        char* mq = !kBf16 && kLast && p.mirror && pc.k1 == p.n_rounds ? p.mirror + (uint64_t)q * kGroupBytes + row_first : nullptr;
        rows([&](int j) {
          unsigned char* sx = own + (uint32_t)j * step;
          const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(sx + cur_off);
          const ulonglong2 cv = *reinterpret_cast<const ulonglong2*>(sx + 2u * plane);
          const ulonglong2 xm = *reinterpret_cast<const ulonglong2*>(cur + (uint32_t)draw[j].x * stride);
          const ulonglong2 o = row_update<kObjective, kFunnel>(p.alpha, noise[j], xv, cv, xm, pivot, __int_as_float(draw[j].y), acc, lacc);
          if (kLast) {
            if (kBf16) *reinterpret_cast<unsigned long long*>(oq + j * row_step) = narrow_bf16x4(o);
            else *reinterpret_cast<ulonglong2*>(oq + j * row_step) = o;
            if (!kBf16 && mq) *reinterpret_cast<ulonglong2*>(mq + j * row_step) = o;
          } else {
            *reinterpret_cast<ulonglong2*>(sx + nxt_off) = kBf16 ? widen_bf16x4(narrow_bf16x4(o)) : o;
          }
        });
      }
      if (kLast && have_next) {  // the centres of this tile have been read for the last time
        const char* cq = p.c + (uint64_t)q_next * kGroupBytes + row_first;
        rows([&](int j) {
          unsigned char* sc = own + 2u * plane + (uint32_t)j * step;
          if (kBf16) cp_async_8(sc, cq + j * row_step);
          else cp_async_16_stream(sc, cq + j * row_step);
        });
      }
      // this thread's shares of the round's sums
      float4 s1;
      float a0, a1, l0, l1;
      unpack2(acc.s1a, s1.x, s1.y);
      unpack2(acc.s1b, s1.z, s1.w);
      unpack2(add2(acc.s2a, acc.s2b), a0, a1);
      unpack2(add2(lacc.la, lacc.lb), l0, l1);
      float2 two = make_float2(a0 + a1, l0 + l1);
      if (p.pre_reduce) {
        for (int off = 16; off >= G; off >>= 1) {
          s1.x += __shfl_xor_sync(0xffffffffu, s1.x, off);
          s1.y += __shfl_xor_sync(0xffffffffu, s1.y, off);
          s1.z += __shfl_xor_sync(0xffffffffu, s1.z, off);
          s1.w += __shfl_xor_sync(0xffffffffu, s1.w, off);
          two.x += __shfl_xor_sync(0xffffffffu, two.x, off);
          two.y += __shfl_xor_sync(0xffffffffu, two.y, off);
        }
        if (lane < G) {
          s_sum[buf * E + warp * G + lane] = s1;
          s_two[buf * E + warp * G + lane] = two;
        }
      } else {
        s_sum[buf * E + tid] = s1;
        s_two[buf * E + tid] = two;
      }
      if (kLast && ahead) {
        cp_async_wait_all();  // the next tile's rows have landed: the barrier publishes them too
        if (kBf16 && have_next) {
          rows([&](int j) {
            unsigned char* sx = own + nxt_off + (uint32_t)j * step;
            unsigned char* sc = own + 2u * plane + (uint32_t)j * step;
            *reinterpret_cast<ulonglong2*>(sx) = widen_bf16x4(*reinterpret_cast<const unsigned long long*>(sx));
            *reinterpret_cast<ulonglong2*>(sc) = widen_bf16x4(*reinterpret_cast<const unsigned long long*>(sc));
          });
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
      // while the others finish: the draws and the noise of the next round, the sums of the previous one
      if (!kLast) {
        next_draws();
        next_noise(q, k + 1);
      } else if (ahead) {
        first_draws(0);
        enter_column(q_next);
        next_noise(q_next, 0);
      }
      if (kFar && last_k >= 0 && warp == turn) add_shares(buf == 0 ? 2u : buf - 1u, last_k);  // (not written again before two more barriers)
      turn = turn + 1 == nwarps ? 0 : turn + 1;
      buf = buf == kBuffers - 1u ? 0 : buf + 1;
      last_k = k;
    };
    for (int k = pc.k0; k + 1 < pc.k1; ++k) run_round(k, std::false_type());
    run_round(pc.k1 - 1, std::true_type());
    base = (base + (uint32_t)(pc.k1 - pc.k0)) & 1u;
    if (pc.k1 < p.n_rounds) {  // this CTA's share of a cut tile is in x_nxt
      __threadfence();
      __syncthreads();
      if (tid == 0) *reinterpret_cast<volatile unsigned int*>(p.cut + blockIdx.x) = 1u;
    }
    if (more && !ahead) {  // the rest of the tile that CTA b - 1 has begun
      mbar_wait(bar, phase, p.error);  // (this piece's last round: its slabs are free)
      phase ^= 1u;
      load_piece(next, base);
    }
    pc = next;
  }
  if (last_k >= 0) {
    mbar_wait(bar, phase, p.error);
    if (warp == turn) add_shares(buf == 0 ? kBuffers - 1u : buf - 1u, last_k);
  }
  if (!p.finalize) return;
  finalize_rounds(p.partials, p.n_rounds, (double)p.inv_M, p.tel, p.slot0, p.ring, p.ticket);
}

}  // namespace netmax
