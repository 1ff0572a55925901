// C-ABI implementation of the NetMax round simulator (see include/netmax.h).
//
// Host side: validation, the 32-bit cumulative-threshold and pull-weight tables, buffer
// layout, launches.  Every step of a round runs in the kernels of netmax_kernels.cuh.
#include "../../include/netmax.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <functional>
#include <future>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <unordered_map>
#include <vector>

#include <cuda_runtime.h>

#include "netmax_plain.cuh"
#include "netmax_instances.h"
#include "netmax_policy.h"

using namespace netmax;

namespace {

thread_local std::string g_error;  // failures of calls that have no context

constexpr int kThreads = 256;
constexpr int64_t kMaxM = 16384;
constexpr int64_t kMaxD = ((int64_t)1 << 30) - 32;  // a padded row stays below 2^32 bytes

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

struct DeviceGuard {
  int prev = -1;
  bool ok = true;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) { prev = -1; }
    if (prev != dev) ok = (cudaSetDevice(dev) == cudaSuccess);
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
};

// Page-locked host memory of a context: the error word that a kernel with a bounded wait raises, the
// mirrors that launches write their telemetry and (small rings) their draws to, and the staging area of
// small read-backs.  Locking pages costs more than a small call, so blocks of destroyed contexts are kept
// for the next ones: at most kPinnedKept of them, the rest are freed.
constexpr size_t kPinnedBytes = (size_t)384 << 10;
constexpr size_t kPinnedKept = 8;
// What a block holds: the error word and netmax_measure's result; the telemetry ring, if it is short
// enough (2,048 rounds); a mirror of the trace ring, if that is small enough; the staging area.
constexpr size_t kPinnedTel = 256, kPinnedTrace = kPinnedTel + ((size_t)32 << 10), kPinnedStaging = kPinnedTrace + ((size_t)64 << 10);
constexpr size_t kStagingBytes = kPinnedBytes - kPinnedStaging;
class PinnedPool {
 public:
  // For the current device, whose context has the number `context`.
  unsigned char* get(int device, uint64_t context) {
    {
      std::lock_guard<std::mutex> lock(mu_);
      for (size_t k = n_kept_; k-- > 0;) {
        if (kept_[k].device != device) continue;
        const Block b = kept_[k];
        kept_[k] = kept_[--n_kept_];
        if (b.context == context) return b.p;  // (else: it went with the context it was locked in)
      }
    }
    void* p = nullptr;
    if (cudaHostAlloc(&p, kPinnedBytes, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    return (unsigned char*)p;
  }
  void put(unsigned char* p, int device, uint64_t context) {  // the caller has waited for everything that writes to it
    {
      std::lock_guard<std::mutex> lock(mu_);
      if (n_kept_ < kPinnedKept) {
        kept_[n_kept_++] = Block{p, device, context};
        return;
      }
    }
    cudaFreeHost(p);
    cudaGetLastError();
  }

 private:
  struct Block {
    unsigned char* p;
    int device;
    uint64_t context;
  };
  std::mutex mu_;
  Block kept_[kPinnedKept];
  size_t n_kept_ = 0;
};
PinnedPool& pinned_pool() {
  static PinnedPool* pool = new PinnedPool();  // never destroyed: contexts may outlive static destructors
  return *pool;
}

// Raises a kernel's limit of dynamic shared memory on the current device, once: the attribute belongs to the kernel in
// the device's context and setting it costs microseconds, so what has been set there is remembered (it is never lowered).
cudaError_t allow_smem(const void* kernel, size_t bytes) {
  struct Limit {
    uint64_t context = 0;
    size_t bytes = 0;
  };
  static std::mutex mu;
  static auto* set = new std::unordered_map<uint64_t, Limit>();
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t key = (uint64_t)(uintptr_t)kernel * 64u + (uint64_t)(dev & 63), context = context_number();
  std::lock_guard<std::mutex> lock(mu);
  Limit& have = (*set)[key];
  if (have.context == context && bytes <= have.bytes) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) {
    have.context = context;
    have.bytes = bytes;
  }
  return e;
}

// Doubles that are not cleared when the vector grows (that would touch every page on one thread).
template <typename T>
struct Uncleared : std::allocator<T> {
  template <typename U>
  struct rebind {
    typedef Uncleared<U> other;
  };
  template <typename U>
  void construct(U* p) {
    ::new ((void*)p) U;
  }
  template <typename U, typename... Args>
  void construct(U* p, Args&&... args) {
    ::new ((void*)p) U(std::forward<Args>(args)...);
  }
};
typedef std::vector<double, Uncleared<double>> HostMatrix;

struct RoundPlan {  // launch shape of round_kernel and multi_round_kernel
  int cg = kThreads, rl = 1, rg = 1, rows_per_group = 0;
  bool short_vectors = false;  // fewer than two streaming tiles per SM: the L2-resident shape
  int grid = 1;
  size_t smem = 0;
  int64_t n_tiles = 0;
};

struct FusedPlan {  // launch shape of fused_rounds_kernel
  bool ok = false;
  int threads = 0, grid = 0, max_rounds = 0;
  int slots = 0;  // rounds the kernel's table of draws is sized for
  size_t smem = 0;
  int64_t n_tiles = 0;
};

struct TilePlan {  // launch shape of tile_rounds_kernel
  bool ok = false;
  int threads = 0, grid = 0, G = 0, log2G = 0, rows = 0;  // rows: per thread
  bool pre_reduce = false;
  size_t smem = 0;
  int64_t n_tiles = 0, max_rounds = 0;
  int64_t min_rounds = 1;  // rounds a call must run to repay loading and storing the tiles
};

struct PipePlan {  // launch shape of pipe_rounds_kernel
  bool ok = false;
  int G = 0, log2G = 0, rows = 0, movers = 0, helpers = 0, batch = 0, grid = 0;
  size_t smem = 0;
  int64_t n_tiles = 0, max_rounds = 0, min_rounds = 0;
};

struct Layout {
  int64_t ld = 0, ldq = 0, nq = 0;  // row stride in elements / in 16-byte column groups; column groups in use
  int elem = 4, halves = 1;         // bytes per stored element; Philox blocks (4 elements) per column group
  size_t plane = 0;                 // bytes of one [M][ld] array
  size_t off_x0 = 0, off_x1 = 0, off_c = 0, off_thr = 0, off_last = 0, off_w = 0, off_trace = 0, off_draws = 0, off_tel = 0,
         off_partials = 0, off_ticket = 0, off_colpart = 0, off_coltick = 0, off_pipe_tel = 0, total = 0;
};

constexpr int kFuseRoundsLimit = 8;  // largest netmax_config.fuse_rounds
constexpr int kMaxGrid = 148 * 16;  // upper bound on resident CTAs of the round kernel
constexpr int64_t kCutLaps = 16, kCutRounds = 16;  // tiles are cut for up to this many tiles per CTA, from this many rounds on
// pipe_rounds_kernel against tile_rounds_kernel (us per call of 64 rounds, tiles / here): 3 x 1,575 elements 58 / 27, 12 x 12,627
// 65 / 49, 48 x 4,735 68 / 56, 96 x 2,367 70 / 63, 128 x 1,183 64 / 68; where the model says 1,600 cycles per round and more
// (3 x 101,031 elements, 64 x 4,735) tiles are as fast or faster.  Calls of four rounds gain 2 to 15 % up to 64
// workers (80: -5 %), of eight 8 to 40 %.
constexpr int kPipeWorkers = 100;
// With more than 36 workers the model knows too little of the telemetry's share from 1,300 cycles on (us per call of 6 and 64 rounds, tiles /
// here, at 1,498: 57 x 3,783 elements 23.3 / 25.1 and 73.7 / 77.1, 56 x 4,719 23.7 / 25.1 and 73.2 / 68.1; 7 x 30,291 24.4 / 22.7 and
// 73.4 / 56.3; at 1,224: 98 x 1,538 23.4 / 23.4 and 74.5 / 60.2).
constexpr double kPipeCycles = 1500.0, kPipeCyclesMany = 1300.0;
constexpr int kPipeMany = 36;
constexpr int64_t kMaxRoundsPerLaunch = 4096;  // rounds one cooperative launch runs at most
constexpr size_t kPartialsBytes = (size_t)kMaxGrid * 2 * sizeof(double) * 8;  // per CTA and round of a fused launch; two sets for multi-round launches
constexpr size_t kColPartBytes = (size_t)8 << 20;  // column partials of the row-split (short vector) shape
constexpr int kMaxChunks = 32;  // column chunks of a pipelined host round trip

Layout make_layout(int64_t M, int64_t d, int64_t trace_rounds, int storage) {
  Layout L;
  L.elem = storage == NETMAX_STORAGE_BF16 ? 2 : 4;
  L.halves = storage == NETMAX_STORAGE_BF16 ? 2 : 1;
  const int64_t per_group = 16 / L.elem;
  L.ld = (int64_t)align_up((size_t)d, (size_t)(128 / L.elem));  // rows start on 128-byte boundaries
  L.ldq = L.ld / per_group;
  L.nq = (d + per_group - 1) / per_group;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 256); return at; };
  const size_t plane = (size_t)M * L.ld * L.elem;
  L.plane = plane;
  L.off_x0 = take(plane);
  L.off_x1 = take(plane);
  L.off_c = take(plane);
  L.off_thr = take((size_t)M * M * sizeof(uint32_t));
  L.off_last = take((size_t)M * sizeof(int32_t));
  L.off_w = take((size_t)M * M * sizeof(float));
  L.off_trace = take((size_t)trace_rounds * M * sizeof(int32_t));
  L.off_draws = take((size_t)trace_rounds * M * sizeof(int2));  // (peer, pull weight) of every draw in the trace ring
  L.off_tel = take((size_t)trace_rounds * 2 * sizeof(double));
  L.off_partials = take(kPartialsBytes);
  L.off_ticket = take(256);
  L.off_colpart = take(kColPartBytes);
  L.off_coltick = take((size_t)kMaxGrid * sizeof(unsigned int));
  L.off_pipe_tel = take((size_t)kMaxChunks * trace_rounds * 2 * sizeof(double));  // per-chunk telemetry of a pipelined round trip
  L.total = o;
  return L;
}

}  // namespace

namespace netmax {
void set_global_error(const std::string& msg) { g_error = msg; }
}  // namespace netmax

struct netmax_ctx {
  int32_t M = 0;
  int64_t d = 0;
  uint32_t q_offset = 0;  // element_offset / 4: added to the column-group word of the counters
  Layout L;
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_memory = false;
  unsigned char* base = nullptr;
  uint64_t context = 0;             // number of the CUDA context that everything below was made in
  unsigned char* pinned = nullptr;  // block of the pinned pool: see kPinnedTel and the rest
  bool host_writes = false;         // launches that may still write to `pinned` have been enqueued since the last synchronisation
  bool read_since_round = false;    // netmax_read_replicas has been called since the last netmax_round
  bool staged = false;              // the staging area holds, or is about to hold, the current replicas
  bool replicas_exposed = false;    // a program may change the replicas behind the library: reads go to the device
  int32_t* trace_mirror = nullptr;  // host copy of the trace ring, written by the sampler (small rings only)
  int storage = NETMAX_STORAGE_F32;
  unsigned char *x[2] = {nullptr, nullptr}, *c = nullptr;  // [M][ld] fp32 or bfloat16, as `storage` says
  uint32_t* thr = nullptr;
  int32_t* last_nz = nullptr;
  float* wtab = nullptr;
  int32_t* trace = nullptr;
  int2* draws = nullptr;  // (peer, bits of the pull weight) of every draw in the trace ring
  // A program that looks at telemetry or peers after every call finds them in page-locked host memory; the writes there
  // cost the launches about 2 us (8 x 524,291 elements: 18.8 us per round, 20.8), so only the rounds of a call that
  // follows such a look go there (and the first call's).  on_host says it for every slot of the rings.
  double *tel_dev = nullptr, *tel_host = nullptr;  // telemetry rings; tel_host only where it is short enough
  double* tel = nullptr;                           // the one of the two that the present call's rounds go to
  bool tel_read = true, trace_read = true;         // looked at since the last call that ran rounds
  bool trace_now = false;                          // the present call's peers go to trace_mirror as well
  std::vector<uint8_t> on_host;                    // [trace_rounds]: 1 telemetry, 2 peers
  double* partials = nullptr;
  unsigned int* ticket = nullptr;
  float4* colpart = nullptr;
  unsigned int* grid_barrier = nullptr;  // arrival counter of multi-round launches
  volatile unsigned int* dev_error = nullptr;  // raised by a kernel whose bounded wait gave up (page-locked host memory)
  bool cooperative = false;              // device supports cooperative launches
  uint32_t inject_absent_ctas = 0;       // test hook: applied to the next multi-round launch, then cleared
  double* measure_out = nullptr;         // (consensus, loss) of netmax_measure (page-locked host memory)
  // host copies of the tables in force (the asynchronous timeline draws peers on the host)
  bool host_tables = false;  // are they those of the policy in force? (need_host_tables)
  std::vector<uint32_t> h_thr;
  std::vector<int32_t> h_last;
  std::vector<float> h_w;
  HostMatrix t_iter;           // iteration times derived from the link speeds in force
  // asynchronous timeline (one worker per global step)
  bool async_on = false;
  double beta = 0.0;
  double now = 0.0;
  int64_t steps = 0;
  std::vector<int64_t> local_n;
  std::vector<int32_t> pending_peer;
  std::vector<float> pending_weight;    // Eq. 16's weight for the pending iteration, under the policy it started with
  std::vector<double> pending_duration; // t_im of the pending iteration, under the times it started with
  std::vector<double> finish;
  // pending iterations ordered by (finish time, worker): exactly one entry per worker
  std::vector<std::pair<double, int>> queue;  // a binary heap, the earliest on top
  std::vector<uint8_t> step_writes, step_reads;  // rows that the launch being put together touches (all 0 between launches)
  std::vector<double> ema;
  std::vector<int64_t> ema_count;
  double monitor_period = 0.0, monitor_next = 0.0;  // Network Monitor on the simulated clock (0: off)
  int64_t monitor_refreshes = 0;
  int64_t ev_cap = 0;
  std::vector<int32_t> ev_worker, ev_peer;
  std::vector<int64_t> ev_n;
  std::vector<double> ev_time;
  unsigned int* coltick = nullptr;
  double* pipe_tel = nullptr;                      // [kMaxChunks][trace_rounds][2]
  cudaStream_t up_stream = nullptr, down_stream = nullptr;  // host round trips: uploads and downloads beside the context's stream
  int cur = 0;  // index of the buffer holding the current replicas
  int64_t rounds = 0;  // number of the next round (absolute)
  int64_t round0 = 0;  // number of the context's first round
  int64_t trace_rounds = 0;
  double alpha = 0, rho = 0, sigma = 0;
  double pull_weight = 0;  // > 0: fixed weight of every pull
  int objective = 1;
  uint64_t seed = 0;
  int policy_K = 20, policy_R = 20;
  double policy_rho_upper = 0.0;
  int fuse_rounds = 0;  // 0: automatic, 1: one launch per round, 2..kFuseRoundsLimit: rounds per fused launch
  bool round_planned[2] = {false, false};  // [0]: the context's objective, [1]: measuring
  RoundPlan round_plan[2];
  bool fused_planned = false;
  FusedPlan fused;
  bool tiles_planned = false;
  TilePlan tiles;
  bool pipe_planned = false;
  PipePlan pipe;
  PhiloxKeys keys;
  DeviceArena arena;          // of changes of links (many workers)
  HostMatrix t_spare;         // the iteration times of new links, worked out while the policy is searched
  std::vector<double> P;      // policy in force
  std::vector<uint8_t> adj;   // link graph in force
  int sm_count = 148;
  int64_t launches = 0;
  std::string error;
};

namespace {

int fail(netmax_ctx* ctx, int code, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  if (ctx) ctx->error = buf; else g_error = buf;
  return code;
}

#define NM_CATCH_CTX(ctx) NM_CATCH([&](int code, const char* what) { return ::fail(ctx, code, "%s", what); })

#define NM_CUDA(ctx, call)                                                                         \
  do {                                                                                             \
    cudaError_t e_ = (call);                                                                       \
    if (e_ != cudaSuccess)                                                                         \
      return fail(ctx, e_ == cudaErrorMemoryAllocation ? NETMAX_OOM : NETMAX_CUDA_ERROR, "%s: %s", \
                  #call, cudaGetErrorString(e_));                                                  \
  } while (0)

// From here on whole M x M matrices are worked on by threads.
constexpr int32_t kManyWorkers = 320;
// From here on Algorithm 3 runs on the device.  ms for a change of links, host / device, K = R = 8: 200 workers 3.9 / 2.4, 256: 5.9 / 2.3,
// 288: 7.3 / 2.2; K = R = 20: 200 workers 7.0 / 7.0 (half the links: 7.0-9.7 / 8.3-9.3), 256: 11.3 / 6.9, 288: 13.9 / 6.2.  A process's
// first change loads the device's kernels, about 6 ms (K = R = 8: 200 workers 5.8 / 9.3, 256: 8 / 10, 288: 10.3 / 9.3): the line lies
// where that one is no slower either.
constexpr int32_t kDevicePolicy = 288;

// Link graph from speeds: d_im = 1 iff i != m and the speed is positive (symmetrised).
int build_adjacency(netmax_ctx* ctx, int32_t M, const double* speed, std::vector<uint8_t>& adj) {
  adj.assign((size_t)M * M, 1);
  std::atomic<int64_t> bad{-1};
  constexpr int64_t kBlock = 64;  // the transposed entries are read a cache line at a time
  parallel_rows(M, kManyWorkers, [&](int64_t r0, int64_t r1) {
    for (int64_t ib = r0; ib < r1; ib += kBlock)
      for (int64_t mb = 0; mb < M; mb += kBlock)
        for (int64_t i = ib; i < std::min(r1, ib + kBlock); ++i)
          for (int64_t m = mb; m < std::min<int64_t>(M, mb + kBlock); ++m) {
            if (i == m) { adj[(size_t)i * M + m] = 0; continue; }
            if (!speed) continue;
            const double a = speed[(size_t)i * M + m], b = speed[(size_t)m * M + i];
            if (!std::isfinite(a)) bad = i * M + m;
            adj[(size_t)i * M + m] = (a > 0.0 && b > 0.0) ? 1 : 0;
          }
  });
  if (bad >= 0) return fail(ctx, NETMAX_INVALID_ARG, "link speed (%d,%d) is not finite", (int)(bad / M), (int)(bad % M));
  // connectivity (Assumption 1) by a depth-first walk from worker 0
  std::vector<int> stack{0};
  std::vector<uint8_t> seen(M, 0);
  seen[0] = 1;
  int count = 1;
  while (!stack.empty() && count < M) {
    const int v = stack.back();
    stack.pop_back();
    for (int m = 0; m < M; ++m)
      if (adj[(size_t)v * M + m] && !seen[m]) { seen[m] = 1; ++count; stack.push_back(m); }
  }
  if (count != M) return fail(ctx, NETMAX_NOT_CONNECTED, "link graph is not connected (%d of %d workers reachable)", count, M);
  return NETMAX_OK;
}

int validate_policy(netmax_ctx* ctx, int32_t M, const double* P, const std::vector<uint8_t>& adj) {
  auto row = [&](int i, bool report) -> int {  // the checks of one row; the message only when asked for
    double sum = 0.0;
    for (int m = 0; m < M; ++m) {
      const double p = P[(size_t)i * M + m];
      if (!(p >= 0.0) || !std::isfinite(p))
        return report ? fail(ctx, NETMAX_BAD_PROB_ROW, "P[%d,%d] = %g is negative or not finite", i, m, p) : NETMAX_BAD_PROB_ROW;
      if (p > 0.0 && m != i && !adj[(size_t)i * M + m])
        return report ? fail(ctx, NETMAX_BAD_PROB_ROW, "P[%d,%d] > 0 on a missing link (Eq. 12)", i, m) : NETMAX_BAD_PROB_ROW;
      sum += p;
    }
    if (std::fabs(sum - 1.0) > 1e-9) return report ? fail(ctx, NETMAX_BAD_PROB_ROW, "row %d of P sums to %.12g", i, sum) : NETMAX_BAD_PROB_ROW;
    return NETMAX_OK;
  };
  std::atomic<int> first_bad{M};
  parallel_rows(M, kManyWorkers, [&](int64_t a, int64_t b) {
    for (int64_t i = a; i < b; ++i)
      if (row((int)i, false) != NETMAX_OK) {
        int seen = first_bad;
        while ((int)i < seen && !first_bad.compare_exchange_weak(seen, (int)i)) {}
        return;
      }
  });
  return first_bad < M ? row(first_bad, true) : NETMAX_OK;
}

// rho <= 0: the largest rho that keeps Eq. 11 (p_im > alpha rho (d_im + d_mi)) with a 1e-6 margin.
double default_rho(int32_t M, const double* P, const std::vector<uint8_t>& adj, double alpha) {
  std::vector<double> row_best(M, INFINITY);
  parallel_rows(M, kManyWorkers, [&](int64_t a, int64_t b) {
    for (int64_t i = a; i < b; ++i) {
      double best = INFINITY;
      for (int64_t m = 0; m < M; ++m) {
        const double p = P[(size_t)i * M + m];
        if (i == m || !(p > 0.0)) continue;
        best = std::min(best, p / (alpha * (2.0 * (double)adj[(size_t)i * M + m])));  // (the graph is symmetric)
      }
      row_best[i] = best;
    }
  });
  const double best = *std::min_element(row_best.begin(), row_best.end());
  return std::isfinite(best) ? (1.0 - 1e-6) * best : 0.0;
}

// A caller's rho must keep Eq. 11, p_im >= alpha rho (d_im + d_mi) on every link in use (taken
// closed, as Algorithm 3's rows may sit on the floor): otherwise the pull weight of Eq. 16
// exceeds 1/2, entries of Y_P (Eq. 22) can turn negative and Theorem 3's lambda_2 < 1 is lost.
// With a fixed pull weight rho is unused and nothing is checked.
int check_rho(netmax_ctx* ctx, int32_t M, const double* P, const std::vector<uint8_t>& adj, double alpha, double rho,
              double pull_weight) {
  if (pull_weight > 0.0) return NETMAX_OK;
  for (int i = 0; i < M; ++i)
    for (int m = 0; m < M; ++m) {
      const double p = P[(size_t)i * M + m];
      if (i == m || !(p > 0.0)) continue;
      const double floor_im = alpha * rho * ((double)adj[(size_t)i * M + m] + (double)adj[(size_t)m * M + i]);
      if (floor_im > p * (1.0 + 1e-9))
        return fail(ctx, NETMAX_INVALID_ARG, "rho = %g breaks Eq. 11 on link (%d,%d): alpha rho (d_im + d_mi) = %g > p_im = %g",
                    rho, i, m, floor_im, p);
    }
  return NETMAX_OK;
}

// T_j = floor(cum_j 2^32 + 1/2) over the left-to-right double prefix sums of the row,
// non-decreasing, saturated, and pinned to the top from the last positive entry on.
void build_tables(int32_t M, const double* P, const std::vector<uint8_t>& adj, double alpha32, double rho,
                  double pull_weight, std::vector<uint32_t>& thr, std::vector<int32_t>& last_nz, std::vector<float>& w) {
  thr.resize((size_t)M * M);
  last_nz.resize(M);
  w.resize((size_t)M * M);
  for (int i = 0; i < M; ++i) {
    const double* p = P + (size_t)i * M;
    int32_t last = -1;
    for (int j = 0; j < M; ++j) if (p[j] > 0.0) last = j;
    last_nz[i] = last;
    double cum = 0.0;
    uint64_t prev = 0;
    for (int j = 0; j < M; ++j) {
      cum += p[j];
      uint64_t t = (uint64_t)std::floor(cum * 4294967296.0 + 0.5);
      t = std::max(t, prev);
      if (t > 0xFFFFFFFFull || j >= last) t = 0xFFFFFFFFull;
      thr[(size_t)i * M + j] = (uint32_t)t;
      prev = t;
      float wv = 0.0f;
      if (j != i && p[j] > 0.0) {
        const double dsum = (double)adj[(size_t)i * M + j] + (double)adj[(size_t)j * M + i];
        wv = pull_weight > 0.0 ? (float)pull_weight                         // fixed-weight averaging
                               : (float)(alpha32 * rho * dsum / (2.0 * p[j]));  // alpha rho gamma_im (Eq. 16)
      }
      w[(size_t)i * M + j] = wv;
    }
  }
}

// Tables from P and the link graph on the device, into the context's own; waits for them (the caller's
// buffers may go).  The asynchronous timeline draws on the host and fetches its copies (need_host_tables).
int device_tables(netmax_ctx* ctx, const double* d_P, const uint8_t* d_adj) {
  NM_CUDA(ctx, build_tables_device(ctx->M, d_P, d_adj, (double)(float)ctx->alpha * ctx->rho, ctx->pull_weight, ctx->thr, ctx->last_nz,
                                   ctx->wtab, ctx->stream));
  ctx->host_tables = false;
  NM_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  return NETMAX_OK;
}

int need_host_tables(netmax_ctx* ctx) {
  if (ctx->host_tables) return NETMAX_OK;
  const size_t MM = (size_t)ctx->M * ctx->M;
  ctx->h_thr.resize(MM);
  ctx->h_last.resize(ctx->M);
  ctx->h_w.resize(MM);
  NM_CUDA(ctx, BulkPool::get().to_host(ctx->h_thr.data(), ctx->thr, MM * sizeof(uint32_t), ctx->device, ctx->stream));
  NM_CUDA(ctx, BulkPool::get().to_host(ctx->h_w.data(), ctx->wtab, MM * sizeof(float), ctx->device, ctx->stream));
  NM_CUDA(ctx, cudaMemcpyAsync(ctx->h_last.data(), ctx->last_nz, ctx->M * sizeof(int32_t), cudaMemcpyDeviceToHost, ctx->stream));
  NM_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  ctx->host_tables = true;
  return NETMAX_OK;
}

// Puts the tables of the policy in force on the device.  Many workers: they are built there, from P (a caller's P set for
// 320 / 400 / 512 / 700 / 1000 workers: 1.77 / 1.85 / 2.54 / 3.07 / 3.57 ms that way, 0.85 / 1.32 / 2.20 / 4.03 / 8.99 with
// tables from the host).
constexpr int32_t kDeviceTables = 600;
int upload_policy(netmax_ctx* ctx) {
  if (ctx->M >= kDeviceTables) {
    const size_t MM = (size_t)ctx->M * ctx->M;
    DeviceArena arena;
    if (arena.begin(DeviceArena::room(MM * sizeof(double)) + MM)) {
      double* d_P = arena.take<double>(MM);
      uint8_t* d_adj = arena.take<uint8_t>(MM);
      NM_CUDA(ctx, BulkPool::get().to_device(d_P, ctx->P.data(), MM * sizeof(double), ctx->device, ctx->stream));
      NM_CUDA(ctx, BulkPool::get().to_device(d_adj, ctx->adj.data(), MM, ctx->device, ctx->stream));
      return device_tables(ctx, d_P, d_adj);
    }
    // (no device memory to spare beside the caller's workspace: on the host, as for few workers)
  }
  std::vector<uint32_t>& thr = ctx->h_thr;
  std::vector<int32_t>& last = ctx->h_last;
  std::vector<float>& w = ctx->h_w;
  build_tables(ctx->M, ctx->P.data(), ctx->adj, (double)(float)ctx->alpha, ctx->rho, ctx->pull_weight, thr, last, w);
  ctx->host_tables = true;
  // pageable sources: the copies are complete (staged) when these calls return
  NM_CUDA(ctx, cudaMemcpyAsync(ctx->thr, thr.data(), thr.size() * sizeof(uint32_t), cudaMemcpyHostToDevice, ctx->stream));
  NM_CUDA(ctx, cudaMemcpyAsync(ctx->last_nz, last.data(), last.size() * sizeof(int32_t), cudaMemcpyHostToDevice, ctx->stream));
  NM_CUDA(ctx, cudaMemcpyAsync(ctx->wtab, w.data(), w.size() * sizeof(float), cudaMemcpyHostToDevice, ctx->stream));
  NM_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  return NETMAX_OK;
}

// Iteration times of the link speeds in force (equal speeds when none were given).
int refresh_iteration_times(netmax_ctx* ctx, const double* speed) {
  const int32_t M = ctx->M;
  std::vector<double> flat;
  if (!speed) {
    flat.assign((size_t)M * M, 1.0);
    speed = flat.data();
  }
  std::vector<uint8_t> adj2((size_t)M * M);
  ctx->t_iter.resize((size_t)M * M);
  int rc = netmax_iteration_times(M, ctx->d, speed, ctx->t_iter.data(), adj2.data());
  if (rc) return fail(ctx, rc, "%s", netmax_last_error(nullptr));
  return NETMAX_OK;
}

// Algorithm 3 on iteration times: on the device for many workers, on the host for fewer and where the device has no memory
// to spare beside the caller's workspace.
int generate_policy(netmax_ctx* ctx, const double* t_iter, double* P, double* rho) {
  int ndev = 0;
  if (ctx->M >= kDevicePolicy) {
    if (cudaGetDeviceCount(&ndev) == cudaSuccess && ctx->device < ndev) {
      DeviceGuard guard(ctx->device);
      DeviceArena arena;
      const int rc = policy_generate_device(ctx->M, t_iter, ctx->adj.data(), ctx->alpha, ctx->policy_K, ctx->policy_R, ctx->policy_rho_upper,
                                            ctx->stream, arena, P, rho, nullptr);
      if (rc != NETMAX_OOM) return rc;
    }
    cudaGetLastError();
  }
  return netmax_policy_generate_ex(ctx->M, t_iter, ctx->adj.data(), ctx->alpha, ctx->policy_K, ctx->policy_R, ctx->policy_rho_upper, P, rho,
                                   nullptr);
}

// Chooses P and rho: the caller's, or Algorithm 3's.  speed == NULL keeps the iteration times
// in force (or, at creation, takes equal speeds).
int resolve_policy(netmax_ctx* ctx, const double* speed, const double* prob, double rho) {
  const int32_t M = ctx->M;
  if (speed || ctx->t_iter.empty()) {
    int rc = refresh_iteration_times(ctx, speed);
    if (rc) return rc;
  }
  if (prob) {
    int rc = validate_policy(ctx, M, prob, ctx->adj);
    if (rc) return rc;
    if (rho > 0.0) {
      rc = check_rho(ctx, M, prob, ctx->adj, ctx->alpha, rho, ctx->pull_weight);
      if (rc) return rc;
    }
    ctx->P.resize((size_t)M * M);
    parallel_copy(ctx->P.data(), prob, (size_t)M * M * sizeof(double));
    ctx->rho = rho > 0.0 ? rho : default_rho(M, prob, ctx->adj, ctx->alpha);
    return NETMAX_OK;
  }
  ctx->P.assign((size_t)M * M, 0.0);
  double rho_sel = 0.0;
  if (ctx->pull_weight > 0.0) {
    // constant pull weight: Algorithm 3 in the form the paper's extension section prescribes (a floor
    // on p_im in rho's place, balanced columns); rho plays no part in the update
    double floor_sel = 0.0;
    int rc = netmax_policy_generate_fixed_weight(M, ctx->t_iter.data(), ctx->adj.data(), ctx->pull_weight, ctx->policy_K,
                                                 ctx->policy_R, ctx->policy_rho_upper, ctx->P.data(), &floor_sel, nullptr);
    if (rc) return fail(ctx, rc, "%s", netmax_last_error(nullptr));
    ctx->rho = rho > 0.0 ? rho : 0.0;
    return NETMAX_OK;
  }
  int rc = generate_policy(ctx, ctx->t_iter.data(), ctx->P.data(), &rho_sel);
  if (rc) return fail(ctx, rc, "%s", netmax_last_error(nullptr));
  if (rho > 0.0) {  // the caller's rho with Algorithm 3's P: it must still respect that P
    rc = check_rho(ctx, M, ctx->P.data(), ctx->adj, ctx->alpha, rho, ctx->pull_weight);
    if (rc) return rc;
  }
  ctx->rho = rho > 0.0 ? rho : rho_sel;
  return NETMAX_OK;
}

int launch_init(netmax_ctx* ctx, unsigned char* dst, double stddev, uint32_t tag) {
  NM_CUDA(ctx, cudaMemsetAsync(dst, 0, ctx->L.plane, ctx->stream));
  if (stddev == 0.0) return NETMAX_OK;
  InitParams p;
  p.dst = reinterpret_cast<float4*>(dst);
  p.ldq = ctx->L.ldq;
  p.nq = ctx->L.nq;
  p.M = ctx->M;
  p.tail = (int32_t)(ctx->d % (4 * ctx->L.halves));
  p.stddev = (float)stddev;
  p.tag = tag;
  p.q_offset = ctx->q_offset;
  p.keys = ctx->keys;
  const int64_t total = (int64_t)ctx->M * ctx->L.nq;
  const int grid = (int)std::min<int64_t>((total + kThreads - 1) / kThreads, (int64_t)ctx->sm_count * 16);
  if (ctx->L.halves == 2) init_normal_kernel<2><<<grid, kThreads, 0, ctx->stream>>>(p);
  else init_normal_kernel<1><<<grid, kThreads, 0, ctx->stream>>>(p);
  ctx->launches += 1;
  NM_CUDA(ctx, cudaGetLastError());
  return NETMAX_OK;
}

int launch_sampler(netmax_ctx* ctx, uint64_t first_round, int64_t n_rounds, int32_t* out, int2* draws, int64_t slot0,
                   int64_t ring) {
  if (n_rounds <= 0) return NETMAX_OK;
  SampleParams p;
  p.thresholds = ctx->thr;
  p.last_nz = ctx->last_nz;
  p.out = out;
  p.draws = draws;
  p.host_out = draws && ctx->trace_now ? ctx->trace_mirror : nullptr;  // (draws into the context's own ring)
  p.wtab = ctx->wtab;
  p.slot0 = slot0;
  p.ring = ring;
  p.first_round = first_round;
  p.n_rounds = n_rounds;
  p.M = ctx->M;
  p.keys = ctx->keys;
  const int64_t M = ctx->M;
  // Rows in shared memory pay where there is much to draw and a row is drawn from often enough to repay reading it
  // whole (us for thresholds through the caches against rows: 4096 x 64 draws 19 / 19, x 128 32 / 22, x 1024 177 / 45;
  // 1024 x 256 17 / 12, x 4096 141 / 43; 256 x 1024 15 / 12).  Four rows per CTA as long as three CTAs share an SM,
  // else two (8192 x 1024: 160 against 109).
  const int rows = sample_smem((uint32_t)M, 4) <= (size_t)75 * 1024 ? 4 : 2;
  const size_t smem = sample_smem((uint32_t)M, rows);
  if (M >= 128 && n_rounds * M >= ((int64_t)1 << 17) && n_rounds * 40 >= M && n_rounds <= (int64_t)1 << 30 && smem <= (size_t)220 * 1024) {
    auto kernel = rows == 4 ? sample_rows_kernel<4> : sample_rows_kernel<2>;
    NM_CUDA(ctx, allow_smem((const void*)kernel, smem));
    const int64_t groups = (M + rows - 1) / rows;
    // rounds are shared out over CTAs as well where the workers alone would not give every SM three of them
    const int64_t splits = std::max<int64_t>(1, std::min<int64_t>(3 * (int64_t)ctx->sm_count / groups, n_rounds / 256));
    const int64_t per_cta = (n_rounds + splits - 1) / splits;
    kernel<<<dim3((unsigned)groups, (unsigned)((n_rounds + per_cta - 1) / per_cta)), kSampleThreads, smem, ctx->stream>>>(
        p, (uint32_t)per_cta);
    ctx->launches += 1;
    NM_CUDA(ctx, cudaGetLastError());
    return NETMAX_OK;
  }
  const int64_t most = std::max<int64_t>(1, (((int64_t)1 << 31) - 1) / M);  // rounds of one launch: its indices are 32 bits wide
  for (int64_t done = 0; done < n_rounds; done += most) {
    p.n_rounds = std::min<int64_t>(most, n_rounds - done);
    p.first_round = first_round + (uint64_t)done;
    p.slot0 = (slot0 + done) % ring;
    const int64_t total = p.n_rounds * M;
    const int grid = (int)std::min<int64_t>((total + kThreads - 1) / kThreads, (int64_t)ctx->sm_count * 32);
    sample_peers_kernel<<<grid, kThreads, 0, ctx->stream>>>(p);
    ctx->launches += 1;
  }
  NM_CUDA(ctx, cudaGetLastError());
  return NETMAX_OK;
}

using RoundKernel = void (*)(const RoundParams);

using StepKernel = void (*)(const StepParams);

// halves: 1 for fp32 state, 2 for bfloat16 state (Philox blocks per 16-byte column group)
template <int kHalves>
StepKernel pick_step_kernel_h(int objective) {
  return objective == 1 ? step_kernel<1, kHalves> : step_kernel<0, kHalves>;
}
StepKernel pick_step_kernel(int objective, int halves) {
  return halves == 2 ? pick_step_kernel_h<2>(objective) : pick_step_kernel_h<1>(objective);
}

template <int kHalves>
RoundKernel pick_kernel_h(int objective, bool short_vectors) {
  if (objective == 2) return short_vectors ? round_kernel<2, 4, kHalves> : round_kernel<2, 1, kHalves>;
  if (short_vectors) return objective == 1 ? round_kernel<1, 4, kHalves> : round_kernel<0, 4, kHalves>;
#ifdef NETMAX_BF16_LONG_RIF
  if (kHalves == 2) return objective == 1 ? round_kernel<1, NETMAX_BF16_LONG_RIF, kHalves> : round_kernel<0, NETMAX_BF16_LONG_RIF, kHalves>;
#endif
  return objective == 1 ? round_kernel<1, 1, kHalves> : round_kernel<0, 1, kHalves>;
}
RoundKernel pick_kernel(int objective, bool short_vectors, int halves) {
  return halves == 2 ? pick_kernel_h<2>(objective, short_vectors) : pick_kernel_h<1>(objective, short_vectors);
}

using MultiRoundKernel = void (*)(const MultiRoundParams);

MultiRoundKernel pick_multi_kernel(int objective, int halves) {
  if (halves == 2) return objective == 1 ? multi_round_kernel<1, 2> : multi_round_kernel<0, 2>;
  return objective == 1 ? multi_round_kernel<1, 1> : multi_round_kernel<0, 1>;
}

// The kernels' noise scale: sigma (at its fp32 rounding, the value the update is defined with)
// times the constant factor sqrt(2 ln 2) of the Box-Muller radius, which the fast normal generator
// leaves out, rounded once to fp32.
float noise_scale(const netmax_ctx* ctx) { return (float)((double)(float)ctx->sigma * kNormalScale); }

// Rounds from r on whose numbers have the same high word: a launch of many rounds works that part of the noise's counters out
// once.
int64_t same_high_word(uint64_t r) { return ((int64_t)1 << 32) - (int64_t)(r & 0xFFFFFFFFull); }

int floor_pow2(int64_t v) {
  int r = 1;
  while ((int64_t)r * 2 <= v) r *= 2;
  return r;
}

// Tile shape.  Long vectors: all M rows x cg column groups, cg the largest power of two
// (<= 256 threads' worth, i.e. 4 KB of a row) that keeps the tile's share of x within 96 KB, so
// that a row fetched for its own update is still in cache when another row pulls it as a peer
// (measured optimum on cfg 2-4: wider tiles stream better until the peer reads start to miss).
// Short vectors (fewer than two such tiles per SM; everything is L2-resident then): 128-byte
// column segments where M allows, no idle row lanes, and the rows split into rg groups so that
// about two CTAs per SM have work.  The same shape serves many workers with vectors of any length:
// beyond 768 rows the 96 KB rule leaves a tile less than 128 bytes of every row, and a stream of
// 64- or 16-byte pieces costs more than peer rows that come from L2 instead of L1 (4096 x 4096
// elements: 135 us per round with 16-byte pieces, 34 with 128-byte pieces and two row groups;
// 1024 x 65536: 250 against 184).
int plan_round_uncached(netmax_ctx* ctx, RoundPlan& plan, int objective) {
  const int64_t M = ctx->M, nq = ctx->L.nq;
  const int64_t target = 2 * (int64_t)ctx->sm_count;  // the short-vector kernel runs 2 CTAs per SM
  int cg = kThreads;
  while (cg > 1 && (int64_t)cg * 16 * M > 96 * 1024) cg >>= 1;
  int rg = 1;
  if ((nq + cg - 1) / cg < 2 * (int64_t)ctx->sm_count || kThreads / cg > M || cg < 8) {
    plan.short_vectors = true;
    // Candidates in order of preference; the score is the number of CTAs with work, up to the target.
    // First among segments of at least 128 bytes only: a narrower one that happens to give more CTAs
    // loses more at the DRAM pins than it wins (8192 x 2048 elements: 144 us per round with 16-byte
    // pieces and 512 CTAs, 50 with 256-byte pieces and 256 CTAs).  With more workers than resident
    // columns can hold, this kernel is the one that runs by default, and 256-byte pieces measured
    // best there (8192 x 2048: 50 against 55 us; 16384 x 1024: 73 against 84).
    static const int wide_first[] = {8, 16, 32, 64, 128, 256};
    static const int wide_first_large[] = {16, 8, 32, 64, 128, 256};
    static const int any_width[] = {8, 4, 2, 16, 32, 64, 128, 256, 1};
    int64_t best_score = -1;
    auto consider = [&](int cand) {
      const int rl = kThreads / cand;
      if (rl > M && cand != kThreads) return;  // row lanes without rows
      const int64_t nct = (nq + cand - 1) / cand;
      int g = (int)std::min<int64_t>(std::min<int64_t>(32, std::max<int64_t>(1, M / rl)), floor_pow2(std::max<int64_t>(1, target / nct)));
      while (g > 1 && (size_t)nct * g * cand * 32 * ctx->L.halves > kColPartBytes) g >>= 1;
      if (nct * g > kMaxGrid) return;
      const int64_t score = std::min<int64_t>(nct * g, target);
      if (score > best_score) {
        best_score = score;
        cg = cand;
        rg = g;
      }
    };
    for (int cand : (M > 4700 ? wide_first_large : wide_first)) consider(cand);
    if (best_score * 20 < target * 17) {  // fewer than 85 % of the CTAs the SMs can hold: narrower pieces may do better
      best_score = -1;
      for (int cand : any_width) consider(cand);
    }
  }
  plan.cg = cg;
  plan.rl = kThreads / cg;
  plan.rg = rg;
  plan.rows_per_group = (int)((M + rg - 1) / rg);
  plan.n_tiles = (nq + cg - 1) / cg * rg;
  plan.smem = align_up((size_t)M * 8, 16) + (plan.rl > 1 ? (size_t)kThreads * 32 * ctx->L.halves : 0) + 64 * sizeof(double);
  RoundKernel k = pick_kernel(objective, plan.short_vectors, ctx->L.halves);
  // (the kernels also hold a little static shared memory, so the opt-in is needed somewhat below 48 KB of dynamic)
  if (plan.smem > 40 * 1024)
    NM_CUDA(ctx, allow_smem((const void*)k, plan.smem));
  int per_sm = 0;
  NM_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kThreads, plan.smem));
  if (per_sm < 1) return fail(ctx, NETMAX_CUDA_ERROR, "round kernel does not fit on an SM (smem %zu)", plan.smem);
  if (plan.short_vectors && ctx->cooperative) {  // the multi-round kernel needs all of its CTAs resident
    MultiRoundKernel mk = pick_multi_kernel(objective == 2 ? 0 : objective, ctx->L.halves);
    if (plan.smem > 40 * 1024)
      NM_CUDA(ctx, allow_smem((const void*)mk, plan.smem));
    int per_sm_multi = 0;
    NM_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm_multi, mk, kThreads, plan.smem));
    per_sm = std::min(per_sm, per_sm_multi);
    if (per_sm < 1) return fail(ctx, NETMAX_CUDA_ERROR, "multi-round kernel does not fit on an SM (smem %zu)", plan.smem);
  }
  plan.grid = (int)std::min<int64_t>(plan.n_tiles, std::min<int64_t>((int64_t)per_sm * ctx->sm_count, kMaxGrid));
  return NETMAX_OK;
}

// The plan depends only on sizes fixed at creation; asking the driver for occupancies again on every
// call took longer than the launches of a small call.
int plan_round(netmax_ctx* ctx, RoundPlan& plan, int objective) {
  const int k = objective == 2 ? 1 : 0;
  if (!ctx->round_planned[k]) {
    RoundPlan fresh;
    int rc = plan_round_uncached(ctx, fresh, objective);
    if (rc) return rc;
    ctx->round_plan[k] = fresh;
    ctx->round_planned[k] = true;
  }
  plan = ctx->round_plan[k];
  return NETMAX_OK;
}

// Launch shape of tile_rounds_kernel: G column groups per tile, W warps per CTA, K rows per thread.  Modelled on
// measurements of every shape for 32 sizes (2 to 4600 workers): a row costs its scheduler 224 cycles and the rest
// of a thread's round as much as a row (so many rows per thread are better than many threads); a round takes at
// least 1,000 cycles and 450 more for every row of a thread, however little else runs; warp counts that four does
// not divide lose 10 %.  An SM holds 12 to 16 warps (by the registers of the instance) as far as its shared memory
// goes.  The shape chosen is within 2 % of the best one on average.
int plan_tiles_uncached(netmax_ctx* ctx, const RoundPlan& plan, const FusedPlan& fused, TilePlan& f) {
  f = TilePlan();
  if (ctx->fuse_rounds == 1 || fused.ok) return NETMAX_OK;
  const int64_t M = ctx->M, nq = (ctx->d + 3) / 4;
  const bool f32 = ctx->storage == NETMAX_STORAGE_F32;
  if (!plan.short_vectors && ctx->fuse_rounds >= 2 && M > 144) return NETMAX_OK;  // (fuse_rounds: see the C header)
  const size_t per_sm = (size_t)228 * 1024, per_cta = (size_t)226 * 1024;  // (227 KB less the static part)
  // Long vectors of fp32 state with up to 88 workers (144 where fused rounds are asked for): telemetry in double across
  // threads, in fp32 over 18 rows at most, as in the shapes that ran them before (88 x 762,603 elements pay 8 to 11 % for
  // another shape than eleven rows per thread).
  const bool wide = !plan.short_vectors && f32 && M <= (ctx->fuse_rounds >= 2 ? 144 : 88);
  double best = 0.0;
  int best_c = 0;
  {
    for (int G = 32, log2G = 5; G >= 1; G >>= 1, --log2G) {
      for (int W = 1; W <= 16; ++W) {
        const int RL = W * 32 / G;
        const int K = (int)((M + RL - 1) / RL);
        if (wide && !tile_wide(K)) continue;
        if (K > kTileMaxRows || (RL > M && W > 1) || W * 32 > tile_max_threads(K)) continue;
        const int warps = tile_max_threads(K) / 32;  // that an SM's registers hold
        bool pre = false;
        size_t smem = tile_smem(M, W * 32, G, false, K);
        const size_t small = tile_smem(M, W * 32, G, true, K);
        const bool may_pre = !wide || 32 / G * K <= 18;  // (the lanes of a warp are added in fp32)
        if (may_pre && (smem > per_cta || (smem > small && per_sm / (smem + 1024) < std::min<size_t>(warps / W, per_sm / (small + 1024))))) {
          pre = true;
          smem = small;
        }
        if (smem > per_cta) continue;
        const int64_t fit = std::min<int64_t>(warps / W, (int64_t)(per_sm / (smem + 1024)));
        if (fit < 1) continue;
        const int64_t n_tiles = (nq + G - 1) / G;
        const int64_t c = std::min<int64_t>(fit, (n_tiles + ctx->sm_count - 1) / ctx->sm_count);
        const double laps = (double)n_tiles / (double)(ctx->sm_count * c);
        const double passes = laps > 8.0 || (laps > 1.0 && plan.short_vectors) ? laps : std::ceil(laps);  // (few tiles are cut)
        const double cycles = passes * std::max((double)((c * W + 3) / 4) * (224.0 * K + 224.0), 1000.0 + 450.0 * K) *
                              (W % 4 != 0 ? 1.1 : 1.0) * (pre ? 1.03 : 1.0);
        if (best == 0.0 || cycles < best * 0.999) {
          best = cycles;
          best_c = (int)c;
          f.threads = W * 32;
          f.G = G;
          f.log2G = log2G;
          f.rows = K;
          f.pre_reduce = pre;
          f.smem = smem;
          f.n_tiles = n_tiles;
        }
      }
    }
  }
  if (best == 0.0) return NETMAX_OK;
  TileKernel k = pick_tile_kernel(ctx->objective, ctx->L.halves, f.rows, f.G, f.threads / 32);
  NM_CUDA(ctx, cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared));
  NM_CUDA(ctx, allow_smem((const void*)k, f.smem));
  int fit = 0;
  NM_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, k, f.threads, f.smem));
  if (fit < 1) return NETMAX_OK;
  f.grid = (int)std::min<int64_t>(f.n_tiles, std::min<int64_t>((int64_t)std::max(best_c, fit) * ctx->sm_count, kMaxGrid));
  f.grid = (int)std::min<int64_t>(f.grid, (int64_t)fit * ctx->sm_count);
  f.max_rounds = std::max<int64_t>(1, std::min<int64_t>(kMaxRoundsPerLaunch, (int64_t)(kColPartBytes / 16) / f.grid));
  if (plan.short_vectors) {
    // A call pays once for bringing its tiles on chip and back -- narrow columns of all M rows, which stream
    // badly -- and then saves on every round.  Rounds from which that paid in measurements (us per round,
    // resident columns against the per-round kernels, calls of 1 / 2 / 4 / many rounds): 4 x 4096 elements
    // 13.4 / 7.0 / 4.1 / 0.9 against 10.3 / 8.2 / 6.0 / 3.8; 4096 x 1024: 57 / 33 / 21 / 9.5 against
    // 29 / 23 / 19 / 16; 4096 x 4096: 219 / 128 / 80 / 33 against 66 / 61 / 58 / 54; 4096 x 16384:
    // 837 / 492 / 310 / 136 against 195 / 192 / 190 / 188.
    const int64_t elements = M * ctx->d;
    f.min_rounds = elements <= ((int64_t)1 << 20) ? 2 : elements <= ((int64_t)1 << 22) ? 6 : elements <= ((int64_t)1 << 24) ? 8 : 16;
  } else if (ctx->fuse_rounds >= 2) {
    f.min_rounds = 2;
    f.max_rounds = std::min<int64_t>(f.max_rounds, ctx->fuse_rounds);
  } else {
    // fp32 state with more than 66 workers: calls of up to eight rounds keep to one launch per round at the worker counts
    // the header names.  That line is older than this kernel: it was drawn where rows split over a cluster of CTAs were no
    // faster.  This kernel is (nine rounds, 93 to 700 workers: 1.5 to 2 times; 64 workers, two to eight rounds: 1.2 to 1.5
    // times), and such calls forgo that.
    static const unsigned char fused_short[22] = {0, 1, 1, 1, 0, 1, 1, 1, 1, 1, 1, 0, 0, 1, 0, 0, 0, 1, 1, 1, 1, 1};  // M = 67 ... 88
    const bool short_calls = M <= 66 || (M <= 88 && fused_short[M - 67]);
    // bfloat16 state: the tiles' narrow pieces are half as long, and the per-round kernel is nearer (one launch per round
    // against tiles, 2 / 4 / 8 / 16 rounds: 40 workers 0.73 / 0.88 / 1.06 / 1.19, 300: 0.72 / 0.87 / 1.02 / 1.19).
    f.min_rounds = !f32 ? 8 : short_calls ? 2 : 9;
  }
  f.ok = true;
  return NETMAX_OK;
}

int plan_tiles(netmax_ctx* ctx, const RoundPlan& plan, const FusedPlan& fused, TilePlan& f) {
  if (!ctx->tiles_planned) {
    TilePlan fresh;
    int rc = plan_tiles_uncached(ctx, plan, fused, fresh);
    if (rc) return rc;
    ctx->tiles = fresh;
    ctx->tiles_planned = true;
  }
  f = ctx->tiles;
  return NETMAX_OK;
}

// Launch shape of pipe_rounds_kernel: G column groups per tile, tiles (moving warps) and helping warps per CTA, rounds per
// batch.  One CTA per SM and one tile per moving warp.  The cycles of a round are modelled on measurements of 2,278 shapes
// (2 to 64 workers, a quarter of a row of 32 column groups to 16 of them per SM): the moving warp's own chain, the SM's
// issue, the chain of a helping warp over its share of a batch, and what every batch costs; the shape chosen is within 1 %
// of the best one on average.
int plan_pipe_uncached(netmax_ctx* ctx, const RoundPlan& plan, PipePlan& f) {
  f = PipePlan();
  if (!plan.short_vectors || ctx->fuse_rounds == 1 || ctx->M > kPipeWorkers) return NETMAX_OK;
  const int64_t M = ctx->M, nq = (ctx->d + 3) / 4;
  double best = 0.0;
  for (int G = 1, log2G = 0; G <= 32; G *= 2, ++log2G) {
    const int rows = (int)((M + 32 / G - 1) / (32 / G));
    if (rows > kPipeMaxRows) continue;
    const int64_t n_tiles = (nq + G - 1) / G, movers = (n_tiles + ctx->sm_count - 1) / ctx->sm_count;
    if (movers > 8) continue;
    for (int share = 1; share <= (int)(16 / movers) - 1; ++share) {  // helping warps per moving warp
      for (int batch : {32, 16, 8, 4, 2}) {
        const size_t smem = pipe_smem(G, rows, (int)movers, batch);
        if (smem > (size_t)226 * 1024) continue;
        const int own = (batch + share - 1) / share, draws = rows <= 2 ? (own + 1) / 2 : own;
        const int sums = ((batch * G + 31) / 32 + share - 1) / share;
        const double helper = (70.0 + draws * (840.0 + 150.0 * rows) + sums * (770.0 + 35.0 * M)) / batch;
        const double cycles = std::max({200.0 + 100.0 * (rows - 1), 95.0 * movers * rows, helper}) + 670.0 / batch;
        if (best == 0.0 || cycles < best * 0.999) {
          best = cycles;
          f.G = G;
          f.log2G = log2G;
          f.rows = rows;
          f.movers = (int)movers;
          f.helpers = share * (int)movers;
          f.batch = batch;
          f.smem = smem;
          f.n_tiles = n_tiles;
        }
      }
    }
  }
  if (best == 0.0 || best > (M > kPipeMany ? kPipeCyclesMany : kPipeCycles)) return NETMAX_OK;
  f.grid = (int)std::min<int64_t>(f.n_tiles, ctx->sm_count);
  NM_CUDA(ctx, allow_smem((const void*)pick_pipe_kernel(ctx->objective, ctx->L.halves, f.rows), f.smem));
  f.max_rounds = std::min<int64_t>(kMaxRoundsPerLaunch, (int64_t)(kColPartBytes / 16) / f.grid);
  f.min_rounds = M <= 64 ? 4 : 8;
  f.ok = true;
  return NETMAX_OK;
}

int plan_pipe(netmax_ctx* ctx, const RoundPlan& plan, PipePlan& f) {
  if (!ctx->pipe_planned) {
    PipePlan fresh;
    int rc = plan_pipe_uncached(ctx, plan, fresh);
    if (rc) return rc;
    ctx->pipe = fresh;
    ctx->pipe_planned = true;
  }
  f = ctx->pipe;
  return NETMAX_OK;
}

int plan_fused_uncached(netmax_ctx* ctx, const RoundPlan& plan, FusedPlan& f) {
  f = FusedPlan();
  if (ctx->fuse_rounds == 1 || plan.short_vectors) return NETMAX_OK;
#ifdef NETMAX_FUSED_MAX_M
  if (ctx->M > NETMAX_FUSED_MAX_M) return NETMAX_OK;
#endif
  const int64_t M = ctx->M;
  // (two and three workers: a round is too short to hide its sums' shuffles, and launches of more than eight rounds lose
  // 1.5 %; four workers: as fast)
  const int want_rounds = ctx->fuse_rounds >= 2 ? std::min(ctx->fuse_rounds, kFusedMaxRounds) : M <= 3 ? 8 : kFusedMaxRounds;
  // 256 or 128 threads per CTA (a multiple of four warps keeps the SM's four schedulers evenly
  // loaded: 3 x 96 threads measured 587 us per cfg3 round against 508 for 2 x 128), whichever
  // puts more threads on an SM with at least two CTAs (one loads its tile while the other
  // computes; M = 16: 1 x 256 threads 529 us).  Every thread needs 48 M bytes of shared memory,
  // and the kernel's ~100 registers cap an SM at 16 warps (capping it at 96 or 80 registers for
  // 18-20 warps measured slower: 135 and 157 us against 128 per cfg2 round).  Beyond 18 workers only
  // 64-thread CTAs fit, three per SM up to M = 24 and two up to M = 36: four to six warps per SM, and
  // faster than one launch per round (M x 4,000,002 elements, us per round, against rows over a cluster of CTAs:
  // M = 20: 132 against 144, 28: 182 against 214, 36: 227 against 287) -- no barrier, no pull that leaves
  // the CTA.  A single such CTA per SM (M = 37 ... 73) is slower (M = 40: 330 against 309), so the kernel is used down to 128 threads per SM.
  for (int rounds : {4, 8, kFusedMaxRounds})
    NM_CUDA(ctx, cudaFuncSetAttribute(pick_fused_kernel(ctx->objective, ctx->L.halves, ctx->M, rounds), cudaFuncAttributePreferredSharedMemoryCarveout,
                                      (int)cudaSharedmemCarveoutMaxShared));
  FusedKernel k = pick_fused_kernel(ctx->objective, ctx->L.halves, ctx->M, 8);  // (the instance with the most registers)
  // The head of the shared memory (draws and telemetry sums) grows with the rounds of a launch: room for as
  // many as were asked for, unless fewer let more threads live on an SM (M = 36: the last kilobytes decide
  // between two CTAs and one).
  int threads = 0, per_sm = 0, slots = 0;
  for (int rounds = want_rounds;; rounds = std::max(2, rounds / 2)) {
    int threads_r = 0, per_sm_r = 0;
    for (int cand : {256, 128, 64}) {
      const size_t smem = fused_head(rounds, M, cand) + (size_t)48 * M * cand;
      if (smem > (size_t)226 * 1024) continue;  // (227 KB less the static part)
      NM_CUDA(ctx, allow_smem((const void*)k, smem));
      int n = 0;
      NM_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, cand, smem));
      if (cand == 64 && per_sm_r >= 2) continue;  // (two-warp CTAs load two of an SM's four schedulers: M = 10, 235 cycles a row against 197)
      const bool better = (n >= 2) != (per_sm_r >= 2) ? n >= 2 : n * cand > per_sm_r * threads_r;
      if (n >= 1 && (threads_r == 0 || better)) { threads_r = cand; per_sm_r = n; }
    }
    if (threads_r != 0 && per_sm_r * threads_r > per_sm * threads) {
      threads = threads_r;
      per_sm = per_sm_r;
      slots = rounds;
    }
    if (rounds <= 4) break;
  }
  if (threads == 0 || per_sm * threads < 128) return NETMAX_OK;  // too few warps to hide the arithmetic latency
  f.threads = threads;
  f.slots = slots;
  f.smem = fused_head(slots, M, threads) + (size_t)48 * M * threads;
  f.max_rounds = slots;
  f.n_tiles = ((ctx->d + 3) / 4 + threads - 1) / threads;
  NM_CUDA(ctx, allow_smem((const void*)k, f.smem));
  f.grid = (int)std::min<int64_t>(f.n_tiles, std::min<int64_t>((int64_t)per_sm * ctx->sm_count, kMaxGrid));
  f.max_rounds = (int)std::min<int64_t>(f.max_rounds, (int64_t)(kPartialsBytes / 16) / f.grid);
  f.ok = true;
  return NETMAX_OK;
}

// Several rounds per launch over shared-memory-resident tiles (fused_rounds_kernel): long
// vectors, fp32 state, and few enough workers that the slabs (48 bytes per worker and thread)
// of at least eight warps fit on an SM.  The plan is kept until fuse_rounds changes.
int plan_fused(netmax_ctx* ctx, const RoundPlan& plan, FusedPlan& f) {
  if (ctx->fused_planned) {
    f = ctx->fused;
    return NETMAX_OK;
  }
  int rc = plan_fused_uncached(ctx, plan, f);
  if (rc == NETMAX_OK) {
    ctx->fused = f;
    ctx->fused_planned = true;
  }
  return rc;
}

// What every launch of the round kernels shares: buffers, tile shape, step sizes, keys.
RoundParams make_round_params(const netmax_ctx* ctx, const RoundPlan& plan) {
  RoundParams p;
  std::memset(&p, 0, sizeof p);
  p.c = reinterpret_cast<const float4*>(ctx->c);
  p.wtab = ctx->wtab;
  p.partials = ctx->partials;
  p.ticket = ctx->ticket;
  p.ldq = ctx->L.ldq;
  p.row_bytes = (uint32_t)(ctx->L.ld * ctx->L.elem);
  p.nq = ctx->L.nq;
  p.n_tiles = plan.n_tiles;
  p.M = ctx->M;
  p.tail = (int32_t)(ctx->d % (4 * ctx->L.halves));
  p.cg = plan.cg;
  p.rl = plan.rl;
  p.rg = plan.rg;
  p.rows_per_group = plan.rows_per_group;
  p.colpart = ctx->colpart;
  p.coltick = ctx->coltick;
  p.alpha = (float)ctx->alpha;
  p.sigma = noise_scale(ctx);
  p.inv_M = 1.0f / (float)ctx->M;
  p.q_offset = ctx->q_offset;
  p.keys = ctx->keys;
  return p;
}

// A range of column groups (four fp32 elements each) of every replica: the whole vector, or one
// chunk of a pipelined host round trip.  Given the draws, columns evolve independently, so the
// kernels run on a range exactly as on the whole: shifted base pointers, the range's group count,
// and the Philox block offset moved along.
struct ColumnRange {
  int64_t q0 = 0, nq4 = 0;  // first group and number of groups (four elements each)
  int32_t tail4 = 0;        // live elements of the range's last group (0: all four); non-zero only at the end of the rows
  bool whole = true;        // the whole vector (the only form bfloat16 state takes)
};

// Launches a kernel that waits for its predecessor itself (wait_for_previous), so that its own start-up runs beside the
// predecessor's end: of the two short kernels of a small call the second one's launch is what is saved.
template <typename Params>
cudaError_t launch_behind_sampler(void (*kernel)(const Params), unsigned grid, int threads, size_t smem, cudaStream_t stream,
                                  const Params& p) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, p);
}

// One launch of tile_rounds_kernel: `chunk` rounds from round r over a column range; the telemetry of its
// rounds is added up by the last CTA (finalize), or by a launch of its own when there are many rounds.
int launch_tiles(netmax_ctx* ctx, cudaStream_t stream, const TilePlan& tiles, const RoundParams& p, const ColumnRange& range,
                 const unsigned char* xin, unsigned char* xout, const unsigned char* cbase, double* tel, uint64_t r, int chunk,
                 bool finalize, unsigned char* mirror) {
  TileParams tp;
  tp.x_cur = reinterpret_cast<const char*>(xin);
  tp.x_nxt = reinterpret_cast<char*>(xout);
  tp.c = reinterpret_cast<const char*>(cbase);
  tp.mirror = reinterpret_cast<char*>(mirror);
  tp.draws = ctx->draws;
  tp.partials = reinterpret_cast<double*>(ctx->colpart);
  tp.tel = tel;
  tp.ticket = ctx->ticket;
  tp.error = const_cast<unsigned int*>(ctx->dev_error);
  tp.slot0 = (int64_t)(r % (uint64_t)ctx->trace_rounds);
  tp.ring = ctx->trace_rounds;
  tp.first_round = r;
  tp.n_rounds = chunk;
  tp.nq = range.nq4;
  tp.n_tiles = (range.nq4 + tiles.G - 1) / tiles.G;
  tp.row_bytes = p.row_bytes;
  tp.M = p.M;
  tp.tail = range.tail4;
  tp.G = tiles.G;
  tp.log2G = tiles.log2G;
  tp.pre_reduce = tiles.pre_reduce ? 1 : 0;
  tp.finalize = finalize ? 1 : 0;
  tp.alpha = p.alpha;
  tp.sigma = p.sigma;
  tp.inv_M = p.inv_M;
  tp.q_offset = ctx->q_offset + (uint32_t)range.q0;
  tp.keys = p.keys;
  TileKernel k = pick_tile_kernel(ctx->objective, ctx->L.halves, tiles.rows, tiles.G, tiles.threads / 32);
  NM_CUDA(ctx, allow_smem((const void*)k, tiles.smem));
  const int64_t grid = std::min<int64_t>(tiles.grid, tp.n_tiles);
  // Few tiles per CTA and enough rounds: equal lengths of cut tiles instead of whole ones, where the last lap
  // would leave more than 3 % of the CTAs' time unused (a cut costs one more load of the tile's rows).
  const int64_t laps = (tp.n_tiles + grid - 1) / grid;
  tp.cut = reinterpret_cast<unsigned int*>(ctx->partials);  // (this kernel keeps its partials in colpart)
  tp.units = 0;
  if (ctx->cooperative && laps >= 2 && laps <= kCutLaps && chunk >= kCutRounds && laps * grid * 100 > tp.n_tiles * 103)
    tp.units = (tp.n_tiles * chunk + grid - 1) / grid;
  if (tp.units > 0) {
    NM_CUDA(ctx, cudaMemsetAsync(tp.cut, 0, (size_t)grid * sizeof(unsigned int), stream));
    void* args[] = {&tp};
    NM_CUDA(ctx, cudaLaunchCooperativeKernel((const void*)k, dim3((unsigned)grid), dim3((unsigned)tiles.threads), args, tiles.smem, stream));
  } else {
    NM_CUDA(ctx, launch_behind_sampler(k, (unsigned)grid, tiles.threads, tiles.smem, stream, tp));
  }
  ctx->launches += 1;
  if (!finalize) {
    const int warps_per_block = kThreads / 32;
    sum_tile_partials_kernel<<<(unsigned)((chunk + warps_per_block - 1) / warps_per_block), kThreads, 0, stream>>>(
        tp.partials, grid, chunk, (double)p.inv_M, tel, tp.slot0, tp.ring);
    ctx->launches += 1;
  }
  NM_CUDA(ctx, cudaGetLastError());
  return NETMAX_OK;
}

// One launch of pipe_rounds_kernel: `chunk` rounds from round r over all columns (see same_high_word).
int launch_pipe(netmax_ctx* ctx, const PipePlan& pipe, const RoundParams& p, const unsigned char* xin, unsigned char* xout,
                uint64_t r, int chunk, unsigned char* mirror) {
  PipeParams pp;
  pp.x_cur = reinterpret_cast<const char*>(xin);
  pp.x_nxt = reinterpret_cast<char*>(xout);
  pp.mirror = reinterpret_cast<char*>(mirror);
  pp.c = reinterpret_cast<const char*>(ctx->c);
  pp.draws = ctx->draws;
  pp.partials = reinterpret_cast<double*>(ctx->colpart);
  pp.slot0 = (int64_t)(r % (uint64_t)ctx->trace_rounds);
  pp.ring = ctx->trace_rounds;
  pp.first_round = r;
  pp.n_rounds = chunk;
  pp.n_tiles = (int32_t)pipe.n_tiles;
  pp.nq = (ctx->d + 3) / 4;
  pp.row_bytes = p.row_bytes;
  pp.M = p.M;
  pp.tail = (int32_t)(ctx->d % 4);
  pp.G = pipe.G;
  pp.log2G = pipe.log2G;
  pp.movers = pipe.movers;
  pp.batch = pipe.batch;
  pp.alpha = p.alpha;
  pp.sigma = p.sigma;
  pp.inv_M = p.inv_M;
  pp.q_offset = ctx->q_offset;
  pp.keys = p.keys;
  PipeKernel k = pick_pipe_kernel(ctx->objective, ctx->L.halves, pipe.rows);
  NM_CUDA(ctx, allow_smem((const void*)k, pipe.smem));
  NM_CUDA(ctx, launch_behind_sampler(k, (unsigned)pipe.grid, (pipe.movers + pipe.helpers) * 32, pipe.smem, ctx->stream, pp));
  const int warps_per_block = kThreads / 32;
  sum_tile_partials_kernel<<<(unsigned)((chunk + warps_per_block - 1) / warps_per_block), kThreads, 0, ctx->stream>>>(
      pp.partials, pipe.grid, chunk, (double)p.inv_M, ctx->tel, pp.slot0, pp.ring);
  ctx->launches += 2;
  NM_CUDA(ctx, cudaGetLastError());
  return NETMAX_OK;
}

// Enqueues rounds [first, first + n) -- their draws are in the trace ring -- for one column range on
// `stream`: many rounds per launch where tiles stay resident (fused_rounds_kernel, or
// tile_rounds_kernel for more workers), else one launch per round.  `cur` is the buffer that holds
// the range's values at round `first`; it is flipped launch by launch.  Telemetry of the range goes
// to tel (ring-indexed like the context's).
int launch_long_rounds(netmax_ctx* ctx, cudaStream_t stream, const RoundPlan& plan, const FusedPlan& fused,
                       const TilePlan& tiles, RoundParams p, const ColumnRange& range, double* tel, uint64_t first,
                       int64_t n, int& cur) {
  RoundKernel kernel = pick_kernel(ctx->objective, plan.short_vectors, ctx->L.halves);
  const size_t shift = range.whole ? 0 : (size_t)range.q0 * 16;  // bytes into every row (fp32 state when not whole)
  const unsigned char* cbase = ctx->c + shift;
  if (!range.whole) {
    p.nq = range.nq4;
    p.n_tiles = (range.nq4 + plan.cg - 1) / plan.cg * plan.rg;
    p.tail = range.tail4;
    p.q_offset = ctx->q_offset + (uint32_t)range.q0;
    p.c = reinterpret_cast<const float4*>(cbase);
  }
  const int round_grid = (int)std::min<int64_t>(plan.grid, p.n_tiles);
  uint64_t r = first;
  for (int64_t b = 0; b < n;) {
    const unsigned char* xin = ctx->x[cur] + shift;
    unsigned char* xout = ctx->x[cur ^ 1] + shift;
    if (tiles.ok && n >= tiles.min_rounds && n - b >= 2) {
      const int64_t launches_left = (n - b + tiles.max_rounds - 1) / tiles.max_rounds;
      const int64_t chunk = std::min((n - b + launches_left - 1) / launches_left, same_high_word(r));
      int rc = launch_tiles(ctx, stream, tiles, p, range, xin, xout, cbase, tel, r, (int)chunk, true, nullptr);
      if (rc) return rc;
      cur ^= 1;
      r += (uint64_t)chunk;
      b += chunk;
      continue;
    }
    if (fused.ok && n - b >= 2) {  // the next rounds in one launch over resident tiles
      // launches of even length (20 rounds at 8 per launch: 7 + 7 + 6, not 8 + 8 + 4)
      const int64_t launches_left = (n - b + fused.max_rounds - 1) / fused.max_rounds;
      const int chunk = (int)std::min((n - b + launches_left - 1) / launches_left, same_high_word(r));
      FusedParams fp;
      fp.x_cur = reinterpret_cast<const float4*>(xin);
      fp.x_nxt = reinterpret_cast<float4*>(xout);
      fp.c = reinterpret_cast<const float4*>(cbase);
      fp.trace = ctx->trace;
      fp.wtab = ctx->wtab;
      fp.tel = tel;
      fp.partials = ctx->partials;
      fp.ticket = ctx->ticket;
      fp.slot0 = (int64_t)(r % (uint64_t)ctx->trace_rounds);
      fp.ring = ctx->trace_rounds;
      fp.first_round = r;
      fp.n_rounds = chunk;
      fp.slots = fused.slots;
      fp.nq = range.nq4;
      fp.n_tiles = (range.nq4 + fused.threads - 1) / fused.threads;
      fp.row_bytes = p.row_bytes;
      fp.M = p.M;
      fp.tail = range.tail4;
      fp.alpha = p.alpha;
      fp.sigma = p.sigma;
      fp.inv_M = p.inv_M;
      fp.q_offset = ctx->q_offset + (uint32_t)range.q0;
      fp.keys = p.keys;
      FusedKernel fk = pick_fused_kernel(ctx->objective, ctx->L.halves, ctx->M, chunk);
      NM_CUDA(ctx, allow_smem((const void*)fk, fused.smem));
      fk<<<(unsigned)std::min<int64_t>(fused.grid, fp.n_tiles), fused.threads, fused.smem, stream>>>(fp);
      ctx->launches += 1;
      cur ^= 1;
      r += (uint64_t)chunk;
      b += chunk;
      continue;
    }
    const int64_t slot = (int64_t)(r % (uint64_t)ctx->trace_rounds);
    p.x_cur = reinterpret_cast<const float4*>(xin);
    p.x_nxt = reinterpret_cast<float4*>(xout);
    p.peers = ctx->trace + slot * ctx->M;
    p.tel_out = tel + 2 * slot;
    p.round_lo = (uint32_t)r;
    p.ctr3 = philox_ctr3(kTagNoise, r);
    if (plan.short_vectors) NM_CUDA(ctx, launch_behind_sampler(kernel, (unsigned)round_grid, kThreads, plan.smem, stream, p));
    else kernel<<<round_grid, kThreads, plan.smem, stream>>>(p);
    ctx->launches += 1;
    cur ^= 1;
    r += 1;
    b += 1;
  }
  NM_CUDA(ctx, cudaGetLastError());
  return NETMAX_OK;
}

}  // namespace

extern "C" {

int netmax_config_init(netmax_config* cfg) {
  if (!cfg) return fail(nullptr, NETMAX_INVALID_ARG, "cfg is NULL");
  std::memset(cfg, 0, sizeof *cfg);
  cfg->objective = 1;
  cfg->trace_rounds = 1024;
  cfg->policy_K = 20;
  cfg->policy_R = 20;
  return NETMAX_OK;
}

static int check_sizes(const netmax_config* cfg) {
  if (!cfg) return fail(nullptr, NETMAX_INVALID_ARG, "cfg is NULL");
  if (cfg->storage != NETMAX_STORAGE_F32 && cfg->storage != NETMAX_STORAGE_BF16)
    return fail(nullptr, NETMAX_INVALID_ARG, "storage = %d is neither NETMAX_STORAGE_F32 nor NETMAX_STORAGE_BF16", cfg->storage);
  if (cfg->storage == NETMAX_STORAGE_BF16 && cfg->element_offset % 8 != 0)
    return fail(nullptr, NETMAX_INVALID_ARG, "element_offset = %lld must be a multiple of 8 with bfloat16 storage", (long long)cfg->element_offset);
  if (cfg->M < 2 || cfg->M > kMaxM) return fail(nullptr, NETMAX_INVALID_ARG, "M = %d outside [2, %lld]", cfg->M, (long long)kMaxM);
  if (cfg->d < 1 || cfg->d >= kMaxD) return fail(nullptr, NETMAX_INVALID_ARG, "d = %lld outside [1, 2^30 - 32)", (long long)cfg->d);
  if (cfg->element_offset < 0 || cfg->element_offset % 4 != 0 || cfg->element_offset + cfg->d >= kMaxD)
    return fail(nullptr, NETMAX_INVALID_ARG, "element_offset = %lld must be a non-negative multiple of 4 with offset + d < 2^30 - 32", (long long)cfg->element_offset);
  if (cfg->trace_rounds < 1) return fail(nullptr, NETMAX_INVALID_ARG, "trace_rounds = %lld < 1", (long long)cfg->trace_rounds);
  if (cfg->fuse_rounds < 0 || cfg->fuse_rounds > kFuseRoundsLimit)
    return fail(nullptr, NETMAX_INVALID_ARG, "fuse_rounds = %d outside [0, %d]", cfg->fuse_rounds, kFuseRoundsLimit);
  if (cfg->first_round < 0 || cfg->first_round >= ((int64_t)1 << 56))
    return fail(nullptr, NETMAX_INVALID_ARG, "first_round = %lld outside [0, 2^56)", (long long)cfg->first_round);
  return NETMAX_OK;
}

int netmax_workspace_size(const netmax_config* cfg, size_t* bytes) {
  int rc = check_sizes(cfg);
  if (rc) return rc;
  if (!bytes) return fail(nullptr, NETMAX_INVALID_ARG, "bytes is NULL");
  *bytes = make_layout(cfg->M, cfg->d, cfg->trace_rounds, cfg->storage).total;
  return NETMAX_OK;
}

int netmax_create_ex(const netmax_config* cfg, netmax_ctx** out) try {
  if (!out) return fail(nullptr, NETMAX_INVALID_ARG, "out is NULL");
  *out = nullptr;
  int rc = check_sizes(cfg);
  if (rc) return rc;
  if (!(cfg->lr > 0.0) || !std::isfinite(cfg->lr)) return fail(nullptr, NETMAX_INVALID_ARG, "lr = %g must be positive and finite", cfg->lr);
  if (!(cfg->sigma >= 0.0) || !std::isfinite(cfg->sigma)) return fail(nullptr, NETMAX_INVALID_ARG, "sigma = %g must be >= 0 and finite", cfg->sigma);
  if (!(cfg->x0_std >= 0.0) || !std::isfinite(cfg->x0_std) || !(cfg->c_std >= 0.0) || !std::isfinite(cfg->c_std))
    return fail(nullptr, NETMAX_INVALID_ARG, "x0_std and c_std must be >= 0 and finite");
  if (!std::isfinite(cfg->rho)) return fail(nullptr, NETMAX_INVALID_ARG, "rho is not finite");
  if (!(cfg->pull_weight >= 0.0 && cfg->pull_weight < 1.0))
    return fail(nullptr, NETMAX_INVALID_ARG, "pull_weight = %g outside [0, 1)", cfg->pull_weight);
  if (cfg->objective != 0 && cfg->objective != 1) return fail(nullptr, NETMAX_INVALID_ARG, "objective = %d is not 0 or 1", cfg->objective);
  if (cfg->device < 0) return fail(nullptr, NETMAX_INVALID_ARG, "device = %d", cfg->device);

  netmax_ctx* ctx = new (std::nothrow) netmax_ctx();
  if (!ctx) return fail(nullptr, NETMAX_OOM, "host allocation failed");
  std::unique_ptr<netmax_ctx, void (*)(netmax_ctx*)> owned(ctx, netmax_destroy);
  auto bail = [&](int code) {
    g_error = ctx->error;
    return code;
  };
  ctx->M = cfg->M;
  ctx->d = cfg->d;
  ctx->q_offset = (uint32_t)(cfg->element_offset / 4);
  ctx->device = cfg->device;
  ctx->stream = (cudaStream_t)cfg->stream;
  ctx->trace_rounds = cfg->trace_rounds;
  ctx->alpha = cfg->lr;
  ctx->sigma = cfg->sigma;
  ctx->pull_weight = cfg->pull_weight;
  ctx->objective = cfg->objective;
  ctx->seed = cfg->seed;
  ctx->policy_K = cfg->policy_K > 0 ? cfg->policy_K : 20;
  ctx->policy_R = cfg->policy_R > 0 ? cfg->policy_R : 20;
  ctx->policy_rho_upper = cfg->policy_rho_upper > 0.0 ? cfg->policy_rho_upper : 0.0;
  ctx->keys = make_philox_keys(cfg->seed);
  ctx->storage = cfg->storage;
  ctx->fuse_rounds = cfg->fuse_rounds;
  ctx->round0 = ctx->rounds = cfg->first_round;
  ctx->L = make_layout(cfg->M, cfg->d, cfg->trace_rounds, cfg->storage);

  rc = build_adjacency(ctx, cfg->M, cfg->link_speed_gbps, ctx->adj);
  if (rc) return bail(rc);
  rc = resolve_policy(ctx, cfg->link_speed_gbps, cfg->prob, cfg->rho);
  if (rc) return bail(rc);

  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
    cudaGetLastError();
    ctx->error = "no CUDA device is available";
    return bail(NETMAX_CUDA_ERROR);
  }
  if (cfg->device >= ndev) { ctx->error = "device ordinal out of range"; return bail(NETMAX_INVALID_ARG); }
  DeviceGuard guard(cfg->device);
  if (!guard.ok) { ctx->error = "cudaSetDevice failed"; return bail(NETMAX_CUDA_ERROR); }
  auto step = [&](cudaError_t e, const char* what) {
    if (e == cudaSuccess) return true;
    ctx->error = std::string(what) + ": " + cudaGetErrorString(e);
    return false;
  };
  int attr = 0;
  if (cudaDeviceGetAttribute(&attr, cudaDevAttrMultiProcessorCount, cfg->device) == cudaSuccess) ctx->sm_count = attr;
  if (cudaDeviceGetAttribute(&attr, cudaDevAttrCooperativeLaunch, cfg->device) == cudaSuccess) ctx->cooperative = attr != 0;
  if (!step(cudaFree(nullptr), "initialising the device")) return bail(NETMAX_CUDA_ERROR);  // (its context, if it is not there yet)
  ctx->context = context_number();
  ctx->pinned = pinned_pool().get(ctx->device, ctx->context);
  if (!ctx->pinned) { ctx->error = "cudaHostAlloc failed"; return bail(NETMAX_OOM); }
  if (cfg->workspace) {
    if (((uintptr_t)cfg->workspace & 255) != 0) { ctx->error = "workspace is not 256-byte aligned"; return bail(NETMAX_INVALID_ARG); }
    if (cfg->workspace_bytes < ctx->L.total) {
      char buf[128];
      snprintf(buf, sizeof buf, "workspace holds %zu bytes, %zu needed", cfg->workspace_bytes, ctx->L.total);
      ctx->error = buf;
      return bail(NETMAX_OOM);
    }
    ctx->base = (unsigned char*)cfg->workspace;
  } else {
    void* ptr = nullptr;
    cudaError_t e = cudaMalloc(&ptr, ctx->L.total);
    if (e != cudaSuccess) {
      cudaGetLastError();
      char buf[160];
      snprintf(buf, sizeof buf, "cudaMalloc of %zu bytes failed: %s", ctx->L.total, cudaGetErrorString(e));
      ctx->error = buf;
      return bail(NETMAX_OOM);
    }
    ctx->base = (unsigned char*)ptr;
    ctx->own_memory = true;
  }
  const Layout& L = ctx->L;
  ctx->x[0] = ctx->base + L.off_x0;
  ctx->x[1] = ctx->base + L.off_x1;
  ctx->c = ctx->base + L.off_c;
  ctx->thr = (uint32_t*)(ctx->base + L.off_thr);
  ctx->last_nz = (int32_t*)(ctx->base + L.off_last);
  ctx->wtab = (float*)(ctx->base + L.off_w);
  ctx->trace = (int32_t*)(ctx->base + L.off_trace);
  ctx->draws = (int2*)(ctx->base + L.off_draws);
  ctx->tel_dev = (double*)(ctx->base + L.off_tel);
  ctx->partials = (double*)(ctx->base + L.off_partials);
  ctx->ticket = (unsigned int*)(ctx->base + L.off_ticket);
  ctx->colpart = (float4*)(ctx->base + L.off_colpart);
  ctx->grid_barrier = ctx->ticket + 16;
  std::memset(ctx->pinned, 0, kPinnedStaging);
  ctx->dev_error = (volatile unsigned int*)ctx->pinned;
  ctx->measure_out = (double*)(ctx->pinned + 64);
  if ((size_t)ctx->trace_rounds * 16 <= kPinnedTrace - kPinnedTel) {
    ctx->tel_host = (double*)(ctx->pinned + kPinnedTel);
  }
  if ((size_t)ctx->trace_rounds * ctx->M * 4 <= kPinnedStaging - kPinnedTrace) ctx->trace_mirror = (int32_t*)(ctx->pinned + kPinnedTrace);
  if (ctx->tel_host || ctx->trace_mirror) ctx->on_host.assign((size_t)ctx->trace_rounds, 0);
  ctx->coltick = (unsigned int*)(ctx->base + L.off_coltick);
  ctx->pipe_tel = (double*)(ctx->base + L.off_pipe_tel);

  if (!step(cudaMemsetAsync(ctx->ticket, 0, 256, ctx->stream), "cudaMemsetAsync(ticket)")) return bail(NETMAX_CUDA_ERROR);
  if (!step(cudaMemsetAsync(ctx->coltick, 0, (size_t)kMaxGrid * sizeof(unsigned int), ctx->stream), "cudaMemsetAsync(coltick)")) return bail(NETMAX_CUDA_ERROR);
  if (!step(cudaMemsetAsync(ctx->x[1], 0, L.plane, ctx->stream), "cudaMemsetAsync(x)")) return bail(NETMAX_CUDA_ERROR);
  if (!step(cudaMemsetAsync(ctx->tel_dev, 0, (size_t)ctx->trace_rounds * 2 * sizeof(double), ctx->stream), "cudaMemsetAsync(tel)")) return bail(NETMAX_CUDA_ERROR);
  rc = upload_policy(ctx);
  if (rc) return bail(rc);
  rc = launch_init(ctx, ctx->x[0], cfg->x0_std, kTagX0);
  if (rc) return bail(rc);
  rc = launch_init(ctx, ctx->c, cfg->c_std, kTagC);
  if (rc) return bail(rc);
  if (!step(cudaStreamSynchronize(ctx->stream), "cudaStreamSynchronize")) return bail(NETMAX_CUDA_ERROR);
  *out = owned.release();
  return NETMAX_OK;
} NM_CATCH_CTX((netmax_ctx*)nullptr)

int netmax_create(int32_t M, int64_t d, const double* link_speed_gbps, const double* prob, double lr, uint64_t seed,
                  netmax_ctx** out) {
  netmax_config cfg;
  netmax_config_init(&cfg);
  cfg.M = M;
  cfg.d = d;
  cfg.link_speed_gbps = link_speed_gbps;
  cfg.prob = prob;
  cfg.lr = lr;
  cfg.seed = seed;
  cfg.x0_std = 1.0;
  cfg.c_std = 1.0;
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cfg.device = dev; else cudaGetLastError();
  return netmax_create_ex(&cfg, out);
}

void netmax_destroy(netmax_ctx* ctx) {
  if (!ctx) return;
  if (ctx->up_stream || ctx->down_stream) {
    DeviceGuard guard(ctx->device);
    if (ctx->up_stream) cudaStreamDestroy(ctx->up_stream);
    if (ctx->down_stream) cudaStreamDestroy(ctx->down_stream);
    cudaGetLastError();
  }
  if (ctx->own_memory && ctx->base) {
    DeviceGuard guard(ctx->device);
    cudaStreamSynchronize(ctx->stream);
    cudaFree(ctx->base);
    cudaGetLastError();
  }
  if (ctx->pinned) {
    if (ctx->host_writes) {  // (the whole device: the caller may have destroyed the stream already)
      DeviceGuard guard(ctx->device);
      cudaDeviceSynchronize();
      cudaGetLastError();
    }
    pinned_pool().put(ctx->pinned, ctx->device, ctx->context);
  }
  delete ctx;
}

// New link speeds and Algorithm 3's policy for them, for many workers: everything that is M x M is worked
// on on the device, from the speeds to the sampler's tables; the host checks the graph meanwhile and keeps
// the iteration times and P.  Nothing of the context changes before the search has succeeded.
static int set_policy_from_links(netmax_ctx* ctx, const double* speed) {
  const int32_t M = ctx->M;
  std::vector<uint8_t> adj;
  std::string graph_error;
  // (a future's destructor waits for its thread, whichever way this function is left; without a thread to be had
  // the work is done at get())
  constexpr auto kBeside = std::launch::async | std::launch::deferred;
  std::future<int> graph = std::async(kBeside, [&] {
    int rc = build_adjacency(nullptr, M, speed, adj);  // (its message goes to this thread's g_error)
    if (!rc) {
      ctx->t_spare.resize((size_t)M * M);
      rc = netmax_iteration_times(M, ctx->d, speed, ctx->t_spare.data(), adj.data());  // (the same graph)
    }
    if (rc) graph_error = g_error;
    return rc;
  });
  ArenaUse use(ctx->arena);
  double* d_P = nullptr;
  uint8_t* d_adj = nullptr;
  double rho = 0.0;
  const int rc = policy_from_links_device(M, ctx->d, speed, ctx->alpha, ctx->policy_K, ctx->policy_R, ctx->policy_rho_upper,
                                          ctx->device, ctx->stream, ctx->arena, &d_P, &d_adj, &rho);
  const int graph_rc = graph.get();
  if (graph_rc) return fail(ctx, graph_rc, "%s", graph_error.c_str());
  if (rc) return fail(ctx, rc, "%s", netmax_last_error(nullptr));
  ctx->rho = rho;
  ctx->t_iter.swap(ctx->t_spare);
  int done = device_tables(ctx, d_P, d_adj);
  if (!done) {
    const cudaError_t e = BulkPool::get().to_host(ctx->P.data(), d_P, (size_t)M * M * sizeof(double), ctx->device, ctx->stream);
    if (e != cudaSuccess) done = fail(ctx, NETMAX_CUDA_ERROR, "reading P back: %s", cudaGetErrorString(e));
  }
  ctx->adj.swap(adj);
  return done;
}

int netmax_set_policy(netmax_ctx* ctx, const double* link_speed_gbps, const double* prob, double rho) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!std::isfinite(rho)) return fail(ctx, NETMAX_INVALID_ARG, "rho is not finite");
  DeviceGuard guard(ctx->device);
  int rc = NETMAX_OK;
  if (ctx->M >= kDevicePolicy && link_speed_gbps && !prob && ctx->pull_weight <= 0.0 && rho <= 0.0) {
    rc = set_policy_from_links(ctx, link_speed_gbps);
    if (!rc && ctx->async_on) rc = need_host_tables(ctx);
    if (rc != NETMAX_OOM) return rc;
    rc = NETMAX_OK;  // (no device memory to spare: piece by piece, as for few workers)
  }
  {
    struct Undo {  // leaves the policy in force untouched unless all of the new one is there
      netmax_ctx* ctx;
      bool links, generated;  // what is replaced: link graph and times; P (a caller's P is checked before it replaces the one in force)
      std::vector<uint8_t> adj;
      std::vector<double> P;
      HostMatrix t;
      double rho;
      bool done = false;
      ~Undo() {
        if (done) return;
        if (links) {
          ctx->adj.swap(adj);
          ctx->t_iter.swap(t);
        }
        if (generated) ctx->P.swap(P);
        ctx->rho = rho;
      }
    };
    std::vector<double> old_P;
    HostMatrix old_t;
    if (!prob) old_P = ctx->P;
    if (link_speed_gbps) old_t = ctx->t_iter;
    Undo undo{ctx, link_speed_gbps != nullptr, prob == nullptr, {}, std::move(old_P), std::move(old_t), ctx->rho};
    if (link_speed_gbps) {
      undo.adj.swap(ctx->adj);
      rc = build_adjacency(ctx, ctx->M, link_speed_gbps, ctx->adj);
    }
    if (!rc) rc = resolve_policy(ctx, link_speed_gbps, prob, rho);
    if (rc) return rc;
    undo.done = true;
  }
  // rounds already enqueued still read the old tables: the new ones are written behind them on the stream
  rc = upload_policy(ctx);
  if (!rc && ctx->async_on) rc = need_host_tables(ctx);
  return rc;
} NM_CATCH_CTX(ctx)

int netmax_get_policy(netmax_ctx* ctx, double* prob_out, double* rho_out) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (prob_out) parallel_copy(prob_out, ctx->P.data(), ctx->P.size() * sizeof(double));
  if (rho_out) *rho_out = ctx->rho;
  return NETMAX_OK;
} NM_CATCH_CTX(ctx)

// Waits for the context's stream; reports a bounded wait of a kernel that has given up since the last check.
static int synchronise(netmax_ctx* ctx) {
  // (an idle stream, as after another read, answers a query sooner than a wait)
  if (cudaStreamQuery(ctx->stream) != cudaSuccess) {
    cudaGetLastError();
    NM_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  }
  ctx->host_writes = false;
  if (*ctx->dev_error == 0u) return NETMAX_OK;
  *ctx->dev_error = 0u;
  return fail(ctx, NETMAX_CUDA_ERROR, "a multi-round launch gave up waiting at a barrier; replicas are not valid");
}

// Copies `bytes` of device memory to the host and synchronises.  Small copies go through the page-locked
// staging area: a copy to pageable memory costs the driver about as much again.
static int read_back(netmax_ctx* ctx, void* host, const void* dev, size_t bytes) {
  const bool staged = bytes <= kStagingBytes;
  unsigned char* stage = ctx->pinned + kPinnedStaging;
  if (staged) ctx->staged = false;
  NM_CUDA(ctx, cudaMemcpyAsync(staged ? stage : host, dev, bytes, cudaMemcpyDeviceToHost, ctx->stream));
  int rc = synchronise(ctx);
  if (rc) return rc;
  if (staged) std::memcpy(host, stage, bytes);
  return NETMAX_OK;
}

// Host transfers of a bfloat16 context go through fp32 on the device: the buffer of the double
// buffer that holds no replicas at the moment serves as the staging area, a chunk of rows at a
// time, and is cleared again afterwards.  Nothing is allocated.
static int64_t staging_rows(const netmax_ctx* ctx) {
  return std::max<int64_t>(1, (int64_t)(ctx->L.plane / ((size_t)ctx->d * sizeof(float))));
}

static int convert_grid(const netmax_ctx* ctx, int64_t total) {
  return (int)std::min<int64_t>((total + kThreads - 1) / kThreads, (int64_t)ctx->sm_count * 16);
}

static int copy_in(netmax_ctx* ctx, unsigned char* dst, const float* host) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!host) return fail(ctx, NETMAX_INVALID_ARG, "host pointer is NULL");
  DeviceGuard guard(ctx->device);
  if (ctx->storage == NETMAX_STORAGE_BF16) {
    float* stage = reinterpret_cast<float*>(ctx->x[ctx->cur ^ 1]);
    const int64_t chunk = staging_rows(ctx);
    for (int64_t r0 = 0; r0 < ctx->M; r0 += chunk) {
      const int64_t rows = std::min<int64_t>(chunk, ctx->M - r0);
      NM_CUDA(ctx, cudaMemcpyAsync(stage, host + (size_t)r0 * ctx->d, (size_t)rows * ctx->d * sizeof(float), cudaMemcpyHostToDevice, ctx->stream));
      narrow_rows_kernel<<<convert_grid(ctx, rows * ctx->d), kThreads, 0, ctx->stream>>>(
          stage, reinterpret_cast<unsigned short*>(dst) + (size_t)r0 * ctx->L.ld, rows, ctx->d, ctx->L.ld);
      ctx->launches += 1;
      NM_CUDA(ctx, cudaGetLastError());
    }
    NM_CUDA(ctx, cudaMemsetAsync(stage, 0, ctx->L.plane, ctx->stream));
    return NETMAX_OK;
  }
  NM_CUDA(ctx, cudaMemcpy2DAsync(dst, (size_t)ctx->L.ld * sizeof(float), host, (size_t)ctx->d * sizeof(float),
                                 (size_t)ctx->d * sizeof(float), (size_t)ctx->M, cudaMemcpyHostToDevice, ctx->stream));
  return NETMAX_OK;
}

static int copy_out(netmax_ctx* ctx, const unsigned char* src, float* host) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!host) return fail(ctx, NETMAX_INVALID_ARG, "host pointer is NULL");
  DeviceGuard guard(ctx->device);
  if (ctx->storage == NETMAX_STORAGE_BF16) {
    float* stage = reinterpret_cast<float*>(ctx->x[ctx->cur ^ 1]);
    const int64_t chunk = staging_rows(ctx);
    for (int64_t r0 = 0; r0 < ctx->M; r0 += chunk) {
      const int64_t rows = std::min<int64_t>(chunk, ctx->M - r0);
      widen_rows_kernel<<<convert_grid(ctx, rows * ctx->d), kThreads, 0, ctx->stream>>>(
          reinterpret_cast<const unsigned short*>(src) + (size_t)r0 * ctx->L.ld, stage, rows, ctx->d, ctx->L.ld);
      ctx->launches += 1;
      NM_CUDA(ctx, cudaGetLastError());
      NM_CUDA(ctx, cudaMemcpyAsync(host + (size_t)r0 * ctx->d, stage, (size_t)rows * ctx->d * sizeof(float), cudaMemcpyDeviceToHost, ctx->stream));
    }
    NM_CUDA(ctx, cudaMemsetAsync(stage, 0, ctx->L.plane, ctx->stream));
    return synchronise(ctx);
  }
  if (ctx->L.ld == ctx->d) return read_back(ctx, host, src, ctx->L.plane);
  if (ctx->L.plane <= kStagingBytes) {  // the padded rows as they are, taken apart on the host
    ctx->staged = false;
    NM_CUDA(ctx, cudaMemcpyAsync(ctx->pinned + kPinnedStaging, src, ctx->L.plane, cudaMemcpyDeviceToHost, ctx->stream));
    int rc = synchronise(ctx);
    if (rc) return rc;
    const float* rows = reinterpret_cast<const float*>(ctx->pinned + kPinnedStaging);
    for (int64_t i = 0; i < ctx->M; ++i) std::memcpy(host + i * ctx->d, rows + i * ctx->L.ld, (size_t)ctx->d * sizeof(float));
    return NETMAX_OK;
  }
  NM_CUDA(ctx, cudaMemcpy2DAsync(host, (size_t)ctx->d * sizeof(float), src, (size_t)ctx->L.ld * sizeof(float),
                                 (size_t)ctx->d * sizeof(float), (size_t)ctx->M, cudaMemcpyDeviceToHost, ctx->stream));
  return synchronise(ctx);
}

int netmax_set_replicas(netmax_ctx* ctx, const float* host_x) {
  if (ctx) ctx->staged = false;
  return copy_in(ctx, ctx ? ctx->x[ctx->cur] : nullptr, host_x);
}
int netmax_set_centres(netmax_ctx* ctx, const float* host_c) { return copy_in(ctx, ctx ? ctx->c : nullptr, host_c); }
int netmax_read_replicas(netmax_ctx* ctx, float* host_out) {
  if (ctx) ctx->read_since_round = true;
  if (ctx && host_out && ctx->staged) {  // on its way since netmax_round; good for one read
    ctx->staged = false;
    DeviceGuard guard(ctx->device);
    const int rc = synchronise(ctx);
    if (rc) return rc;
    const float* rows = reinterpret_cast<const float*>(ctx->pinned + kPinnedStaging);
    for (int64_t i = 0; i < ctx->M; ++i) std::memcpy(host_out + i * ctx->d, rows + i * ctx->L.ld, (size_t)ctx->d * sizeof(float));
    return NETMAX_OK;
  }
  return copy_out(ctx, ctx ? ctx->x[ctx->cur] : nullptr, host_out);
}
int netmax_read_centres(netmax_ctx* ctx, float* host_out) { return copy_out(ctx, ctx ? ctx->c : nullptr, host_out); }

// Where the telemetry and the peers of the n rounds that follow go (see on_host).
static void choose_rings(netmax_ctx* ctx, int64_t n) {
  const bool tel = ctx->tel_host && ctx->tel_read;
  ctx->trace_now = ctx->trace_mirror && ctx->trace_read;
  ctx->tel = tel ? ctx->tel_host : ctx->tel_dev;
  ctx->tel_read = ctx->trace_read = false;
  if (ctx->on_host.empty()) return;
  const uint8_t mark = (uint8_t)((tel ? 1 : 0) | (ctx->trace_now ? 2 : 0));
  const int64_t ring = ctx->trace_rounds, count = std::min(n, ring), at = (ctx->rounds + n - count) % ring, first = std::min(count, ring - at);
  std::memset(ctx->on_host.data() + at, mark, (size_t)first);
  std::memset(ctx->on_host.data(), mark, (size_t)(count - first));
}

// All plans of a context, made by its first call: they ask for their kernels, and with the first one of a family its module is loaded (planning
// only what the call at hand may take put that into later, longer calls).
static int plan_call(netmax_ctx* ctx, const RoundPlan& plan, PipePlan& pipe, FusedPlan& fused, TilePlan& tiles) {
  int rc = plan_fused(ctx, plan, fused);
  if (!rc) rc = plan_tiles(ctx, plan, fused, tiles);
  if (!rc) rc = plan_pipe(ctx, plan, pipe);
  return rc;
}

// Which kernel a batch of rounds takes.
static int batch_kernel(const netmax_ctx* ctx, const RoundPlan& plan, const PipePlan& pipe, const FusedPlan& fused, const TilePlan& tiles, int64_t batch) {
  if (pipe.ok && batch >= pipe.min_rounds) return NETMAX_KERNEL_PIPE;
  if (tiles.ok && batch >= tiles.min_rounds) return NETMAX_KERNEL_TILES;
  if (plan.short_vectors && ctx->cooperative && batch >= 2) return NETMAX_KERNEL_MULTI_ROUND;
  if (fused.ok && batch >= 2) return NETMAX_KERNEL_FUSED;
  return NETMAX_KERNEL_ROUND;
}

int netmax_round(netmax_ctx* ctx, int64_t n_rounds) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (n_rounds < 0) return fail(ctx, NETMAX_INVALID_ARG, "n_rounds = %lld < 0", (long long)n_rounds);
  if (ctx->async_on) return fail(ctx, NETMAX_INVALID_ARG, "the context runs the asynchronous timeline; use netmax_async_steps");
  if (n_rounds == 0) return NETMAX_OK;
  if ((uint64_t)(ctx->rounds + n_rounds) >= ((uint64_t)1 << 56)) return fail(ctx, NETMAX_INVALID_ARG, "round counter would exceed 2^56");
  DeviceGuard guard(ctx->device);
  RoundPlan plan;
  int rc = plan_round(ctx, plan, ctx->objective);
  if (rc) return rc;
  ctx->host_writes = true;
  ctx->staged = false;
  PipePlan pipe;
  FusedPlan fused;
  TilePlan tiles;
  rc = plan_call(ctx, plan, pipe, fused, tiles);
  if (rc) return rc;

  choose_rings(ctx, n_rounds);
  RoundParams p = make_round_params(ctx, plan);

  // A program that reads small replicas after every call gets them with the rounds: the last launch writes them to
  // the page-locked staging area as well (4 x 4096 elements: a copy and a wait of their own were 15 of 45 us).
  unsigned char* mirror = ctx->read_since_round && !ctx->replicas_exposed && ctx->storage == NETMAX_STORAGE_F32 && ctx->L.plane <= kStagingBytes
                              ? ctx->pinned + kPinnedStaging : nullptr;
  bool mirrored = false;
  int64_t done = 0;
  while (done < n_rounds) {
    // peers of a batch of rounds in one launch (counter-based draws do not depend on x),
    // at most one lap of the ring at a time
    const int64_t batch = std::min<int64_t>(n_rounds - done, ctx->trace_rounds);
    rc = launch_sampler(ctx, (uint64_t)ctx->rounds, batch, ctx->trace, ctx->draws, ctx->rounds % ctx->trace_rounds,
                        ctx->trace_rounds);
    if (rc) return rc;
    const int kernel = batch_kernel(ctx, plan, pipe, fused, tiles, batch);
    if (kernel == NETMAX_KERNEL_PIPE) {
      for (int64_t b = 0; b < batch;) {
        const int64_t chunk = std::min({batch - b, pipe.max_rounds, same_high_word((uint64_t)ctx->rounds)});
        rc = launch_pipe(ctx, pipe, p, ctx->x[ctx->cur], ctx->x[ctx->cur ^ 1], (uint64_t)ctx->rounds, (int)chunk,
                         done + b + chunk == n_rounds ? mirror : nullptr);
        if (rc) return rc;
        mirrored = true;
        ctx->cur ^= 1;
        ctx->rounds += chunk;
        b += chunk;
      }
      done += batch;
      continue;
    }
    if (plan.short_vectors && kernel == NETMAX_KERNEL_TILES) {
      // short vectors: every round of the batch on shared-memory-resident columns
      ColumnRange all;
      all.nq4 = (ctx->d + 3) / 4;
      all.tail4 = (int32_t)(ctx->d % 4);
      for (int64_t b = 0; b < batch;) {
        const int64_t chunk = std::min({batch - b, tiles.max_rounds, same_high_word((uint64_t)ctx->rounds)});
        rc = launch_tiles(ctx, ctx->stream, tiles, p, all, ctx->x[ctx->cur], ctx->x[ctx->cur ^ 1], ctx->c, ctx->tel,
                          (uint64_t)ctx->rounds, (int)chunk, false, done + b + chunk == n_rounds ? mirror : nullptr);
        if (rc) return rc;
        mirrored = true;
        ctx->cur ^= 1;
        ctx->rounds += chunk;
        b += chunk;
      }
      done += batch;
      continue;
    }
    if (kernel == NETMAX_KERNEL_MULTI_ROUND) {
      // short, L2-resident problem: all rounds of the batch in cooperative launches
      int64_t b = 0;
      while (b < batch) {
        const int64_t chunk = std::min<int64_t>(batch - b, kMaxRoundsPerLaunch);
        MultiRoundParams mp;
        mp.r = p;
        mp.r.x_cur = reinterpret_cast<const float4*>(ctx->x[ctx->cur]);
        mp.r.x_nxt = reinterpret_cast<float4*>(ctx->x[ctx->cur ^ 1]);
        mp.r.peers = nullptr;
        mp.r.tel_out = nullptr;
        mp.trace = ctx->trace;
        mp.tel = ctx->tel;
        mp.partials2 = ctx->partials;
        mp.barrier = ctx->grid_barrier;
        mp.error = const_cast<unsigned int*>(ctx->dev_error);
        mp.slot0 = ctx->rounds % ctx->trace_rounds;
        mp.ring = ctx->trace_rounds;
        mp.first_round = (uint64_t)ctx->rounds;
        mp.n_rounds = (int32_t)chunk;
        mp.absent_ctas = ctx->inject_absent_ctas;
        ctx->inject_absent_ctas = 0;
        NM_CUDA(ctx, cudaMemsetAsync(ctx->grid_barrier, 0, sizeof(unsigned int), ctx->stream));
        void* args[] = {&mp};
        NM_CUDA(ctx, cudaLaunchCooperativeKernel((const void*)pick_multi_kernel(ctx->objective, ctx->L.halves), dim3(plan.grid), dim3(kThreads),
                                                 args, plan.smem, ctx->stream));
        ctx->launches += 1;
        ctx->cur ^= (int)(chunk & 1);
        ctx->rounds += chunk;
        b += chunk;
      }
      done += batch;
      continue;
    }
    {  // long vectors: resident tiles or one launch per round, over all columns
      ColumnRange all;
      all.q0 = 0;
      all.nq4 = (ctx->d + 3) / 4;
      all.tail4 = (int32_t)(ctx->d % 4);
      all.whole = true;
      int cur = ctx->cur;
      // (the short-vector kernel mirrors a batch of one round; it is the only one that runs here on so few elements)
      const bool one = plan.short_vectors && batch == 1 && done + batch == n_rounds;
      p.mirror = one ? reinterpret_cast<char*>(mirror) : nullptr;
      mirrored = one;
      rc = launch_long_rounds(ctx, ctx->stream, plan, fused, tiles, p, all, ctx->tel, (uint64_t)ctx->rounds, batch, cur);
      if (rc) return rc;
      ctx->cur = cur;
      ctx->rounds += batch;
    }
    NM_CUDA(ctx, cudaGetLastError());
    done += batch;
  }
  ctx->staged = mirror != nullptr && mirrored;
  ctx->read_since_round = false;
  return NETMAX_OK;
} NM_CATCH_CTX(ctx)

int64_t netmax_rounds_done(const netmax_ctx* ctx) { return ctx ? ctx->rounds : -1; }

// ---- host round trip, pipelined over column chunks ----------------------------------------------
int netmax_round_from_host(netmax_ctx* ctx, const float* host_x, const float* host_c, int64_t n_rounds, float* host_out,
                           int32_t n_chunks) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (n_rounds < 0) return fail(ctx, NETMAX_INVALID_ARG, "n_rounds = %lld < 0", (long long)n_rounds);
  if (!host_out) return fail(ctx, NETMAX_INVALID_ARG, "host_out is NULL");
  if (n_chunks < 0 || n_chunks > kMaxChunks) return fail(ctx, NETMAX_INVALID_ARG, "n_chunks = %d outside [0, %d]", n_chunks, kMaxChunks);
  if (ctx->async_on) return fail(ctx, NETMAX_INVALID_ARG, "the context runs the asynchronous timeline; use netmax_async_steps");
  DeviceGuard guard(ctx->device);
  RoundPlan plan;
  int rc = plan_round(ctx, plan, ctx->objective);
  if (rc) return rc;
  const int64_t nq4 = (ctx->d + 3) / 4;
  const int64_t unit = 256;  // chunk boundaries on 4 KB of every row
  // More chunks hide more of the first upload and the last download, but every chunk has launches and copies of its own
  // (upload of 12.8 MB: 0.37 ms with two, 0.43 with eight; 128 MB: 2.86 with four, 2.88 with eight; 715 MB: 15.1 / 14.6).
  const int64_t upload = 8 * (int64_t)ctx->M * ctx->d;
  int chunks = n_chunks > 0 ? n_chunks : upload <= ((int64_t)20 << 20) ? 2 : upload <= ((int64_t)200 << 20) ? 4 : 8;
  chunks = (int)std::min<int64_t>(chunks, (nq4 + unit - 1) / unit);
  const bool pipelined = ctx->storage == NETMAX_STORAGE_F32 && !plan.short_vectors && n_rounds >= 1 &&
                         n_rounds <= ctx->trace_rounds && chunks >= 2 &&
                         (uint64_t)(ctx->rounds + n_rounds) < ((uint64_t)1 << 56);
  if (!pipelined) {  // the same three steps one after the other
    if (host_x) { rc = netmax_set_replicas(ctx, host_x); if (rc) return rc; }
    if (host_c) { rc = netmax_set_centres(ctx, host_c); if (rc) return rc; }
    rc = netmax_round(ctx, n_rounds);
    if (rc) return rc;
    return netmax_read_replicas(ctx, host_out);
  }
  FusedPlan fused;
  rc = plan_fused(ctx, plan, fused);
  if (rc) return rc;
  TilePlan tiles;
  rc = plan_tiles(ctx, plan, fused, tiles);
  if (rc) return rc;
  if (!ctx->up_stream) NM_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->up_stream, cudaStreamNonBlocking));
  if (!ctx->down_stream) NM_CUDA(ctx, cudaStreamCreateWithFlags(&ctx->down_stream, cudaStreamNonBlocking));

  const int64_t per_chunk = ((nq4 + chunks - 1) / chunks + unit - 1) / unit * unit;
  chunks = (int)((nq4 + per_chunk - 1) / per_chunk);
  std::vector<cudaEvent_t> events(2 * chunks + 1, nullptr);
  auto cleanup = [&]() {
    for (cudaEvent_t e : events)
      if (e) cudaEventDestroy(e);
  };
  for (auto& e : events) {
    cudaError_t ce = cudaEventCreateWithFlags(&e, cudaEventDisableTiming);
    if (ce != cudaSuccess) { cleanup(); return fail(ctx, NETMAX_CUDA_ERROR, "cudaEventCreate: %s", cudaGetErrorString(ce)); }
  }
  // from here on a failure still has to wait for what is in flight before the events go away
  auto bail = [&](int code) {
    cudaStreamSynchronize(ctx->up_stream);
    cudaStreamSynchronize(ctx->stream);
    cudaStreamSynchronize(ctx->down_stream);
    cleanup();
    return code;
  };
#define NM_PIPE(call)                                                                                   \
  do {                                                                                                  \
    cudaError_t e_ = (call);                                                                            \
    if (e_ != cudaSuccess) return bail(fail(ctx, NETMAX_CUDA_ERROR, "%s: %s", #call, cudaGetErrorString(e_))); \
  } while (0)

  const uint64_t first = (uint64_t)ctx->rounds;
  choose_rings(ctx, n_rounds);
  ctx->host_writes = true;
  ctx->staged = false;
  rc = launch_sampler(ctx, first, n_rounds, ctx->trace, ctx->draws, ctx->rounds % ctx->trace_rounds, ctx->trace_rounds);
  if (rc) return bail(rc);
  // uploads must not overtake earlier work of the context that still reads the buffers
  NM_PIPE(cudaEventRecord(events[2 * chunks], ctx->stream));
  NM_PIPE(cudaStreamWaitEvent(ctx->up_stream, events[2 * chunks], 0));
  const RoundParams p = make_round_params(ctx, plan);
  const size_t dev_pitch = (size_t)ctx->L.ld * sizeof(float), host_pitch = (size_t)ctx->d * sizeof(float);
  int cur_end = ctx->cur;
  for (int k = 0; k < chunks; ++k) {
    ColumnRange range;
    range.q0 = (int64_t)k * per_chunk;
    range.nq4 = std::min<int64_t>(per_chunk, nq4 - range.q0);
    range.tail4 = (k == chunks - 1) ? (int32_t)(ctx->d % 4) : 0;
    range.whole = false;
    const int64_t e0 = range.q0 * 4, cols = std::min<int64_t>(range.nq4 * 4, ctx->d - e0);
    const size_t width = (size_t)cols * sizeof(float), at = (size_t)e0 * sizeof(float);
    if (host_x)
      NM_PIPE(cudaMemcpy2DAsync(ctx->x[ctx->cur] + at, dev_pitch, host_x + e0, host_pitch, width, (size_t)ctx->M,
                                cudaMemcpyHostToDevice, ctx->up_stream));
    if (host_c)
      NM_PIPE(cudaMemcpy2DAsync(ctx->c + at, dev_pitch, host_c + e0, host_pitch, width, (size_t)ctx->M, cudaMemcpyHostToDevice,
                                ctx->up_stream));
    NM_PIPE(cudaEventRecord(events[2 * k], ctx->up_stream));
    NM_PIPE(cudaStreamWaitEvent(ctx->stream, events[2 * k], 0));
    int cur = ctx->cur;
    rc = launch_long_rounds(ctx, ctx->stream, plan, fused, tiles, p, range, ctx->pipe_tel + (size_t)k * ctx->trace_rounds * 2,
                            first, n_rounds, cur);
    if (rc) return bail(rc);
    cur_end = cur;
    NM_PIPE(cudaEventRecord(events[2 * k + 1], ctx->stream));
    NM_PIPE(cudaStreamWaitEvent(ctx->down_stream, events[2 * k + 1], 0));
    NM_PIPE(cudaMemcpy2DAsync(host_out + e0, host_pitch, ctx->x[cur_end] + at, dev_pitch, width, (size_t)ctx->M,
                              cudaMemcpyDeviceToHost, ctx->down_stream));
  }
  // the rounds' telemetry: the chunks' shares added in chunk order
  sum_chunk_telemetry_kernel<<<(unsigned)((n_rounds + kThreads - 1) / kThreads), kThreads, 0, ctx->stream>>>(
      ctx->pipe_tel, chunks, ctx->trace_rounds, (int64_t)(first % (uint64_t)ctx->trace_rounds), n_rounds, ctx->tel);
  ctx->launches += 1;
  NM_PIPE(cudaGetLastError());
  ctx->cur = cur_end;
  ctx->rounds += n_rounds;
  NM_PIPE(cudaStreamSynchronize(ctx->down_stream));
#undef NM_PIPE
  rc = synchronise(ctx);
  cleanup();
  return rc;
} NM_CATCH_CTX(ctx)

int netmax_set_fuse_rounds(netmax_ctx* ctx, int32_t fuse_rounds) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (fuse_rounds < 0 || fuse_rounds > kFuseRoundsLimit)
    return fail(ctx, NETMAX_INVALID_ARG, "fuse_rounds = %d outside [0, %d]", fuse_rounds, kFuseRoundsLimit);
  ctx->fuse_rounds = fuse_rounds;
  ctx->fused_planned = false;
  ctx->tiles_planned = false;
  ctx->pipe_planned = false;
  return NETMAX_OK;
}

int netmax_read_columns(netmax_ctx* ctx, const int64_t* host_cols, int64_t n_cols, float* host_out) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (n_cols < 0 || (n_cols > 0 && (!host_cols || !host_out))) return fail(ctx, NETMAX_INVALID_ARG, "bad column list");
  if (n_cols == 0) return NETMAX_OK;
  for (int64_t k = 0; k < n_cols; ++k)
    if (host_cols[k] < 0 || host_cols[k] >= ctx->d) return fail(ctx, NETMAX_INVALID_ARG, "cols[%lld] = %lld outside [0, d)", (long long)k, (long long)host_cols[k]);
  DeviceGuard guard(ctx->device);
  int64_t* d_cols = nullptr;
  float* d_out = nullptr;
  NM_CUDA(ctx, cudaMalloc(&d_cols, (size_t)n_cols * sizeof(int64_t)));
  cudaError_t e = cudaMalloc(&d_out, (size_t)n_cols * ctx->M * sizeof(float));
  if (e != cudaSuccess) { cudaFree(d_cols); cudaGetLastError(); return fail(ctx, NETMAX_OOM, "cudaMalloc failed: %s", cudaGetErrorString(e)); }
  int rc = NETMAX_OK;
  const int64_t total = n_cols * ctx->M;
  const int grid = (int)std::min<int64_t>((total + kThreads - 1) / kThreads, 4096);
  e = cudaMemcpyAsync(d_cols, host_cols, (size_t)n_cols * sizeof(int64_t), cudaMemcpyHostToDevice, ctx->stream);
  if (e == cudaSuccess) {
    gather_columns_kernel<<<grid, kThreads, 0, ctx->stream>>>(ctx->x[ctx->cur], ctx->storage == NETMAX_STORAGE_BF16, ctx->L.ld, ctx->M, d_cols, n_cols, d_out);
    ctx->launches += 1;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(host_out, d_out, (size_t)total * sizeof(float), cudaMemcpyDeviceToHost, ctx->stream);
  if (e != cudaSuccess) rc = fail(ctx, NETMAX_CUDA_ERROR, "read_columns: %s", cudaGetErrorString(e));
  const int rs = synchronise(ctx);
  cudaFree(d_cols);
  cudaFree(d_out);
  return rc ? rc : rs;
}

// ---- sampled read-back that allocates nothing -------------------------------------------
// Staging area of netmax_read_columns_static: the column list, then the gathered values.
// It is part of the library image, so every device that loads the library holds it.
struct StaticGatherScratch {
  int64_t cols[NETMAX_STATIC_MAX_COLS];
  float values[NETMAX_STATIC_MAX_VALUES];
};
static __device__ __align__(256) unsigned char g_gather_scratch[sizeof(StaticGatherScratch)];

// In host code g_gather_scratch is only a stand-in for the symbol; the address a kernel or a
// copy can use comes from cudaGetSymbolAddress, looked up once per device and CUDA context (that
// device current) and cached here.
static std::mutex g_gather_mu;
static StaticGatherScratch* g_gather_ptr[64] = {};
static uint64_t g_gather_context[64] = {};

static int gather_scratch_address(netmax_ctx* ctx, StaticGatherScratch** out) {
  std::lock_guard<std::mutex> lock(g_gather_mu);
  const bool cached = ctx->device >= 0 && ctx->device < 64;
  if (cached && g_gather_ptr[ctx->device] && g_gather_context[ctx->device] == ctx->context) {
    *out = g_gather_ptr[ctx->device];
    return NETMAX_OK;
  }
  void* ptr = nullptr;
  NM_CUDA(ctx, cudaGetSymbolAddress(&ptr, g_gather_scratch));
  if (!ptr) return fail(ctx, NETMAX_CUDA_ERROR, "cudaGetSymbolAddress returned a null address");
  if (cached) {
    g_gather_ptr[ctx->device] = (StaticGatherScratch*)ptr;
    g_gather_context[ctx->device] = ctx->context;
  }
  *out = (StaticGatherScratch*)ptr;
  return NETMAX_OK;
}

int netmax_read_columns_static(netmax_ctx* ctx, const int64_t* host_cols, int64_t n_cols, float* host_out) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (n_cols < 0 || (n_cols > 0 && (!host_cols || !host_out))) return fail(ctx, NETMAX_INVALID_ARG, "bad column list");
  if (n_cols > NETMAX_STATIC_MAX_COLS)
    return fail(ctx, NETMAX_INVALID_ARG, "read_columns_static: n_cols = %lld exceeds the fixed staging area (%d columns); split the list",
                (long long)n_cols, NETMAX_STATIC_MAX_COLS);
  if (n_cols * (int64_t)ctx->M > NETMAX_STATIC_MAX_VALUES)
    return fail(ctx, NETMAX_INVALID_ARG, "read_columns_static: M * n_cols = %lld exceeds the fixed staging area (%d values); split the list",
                (long long)(n_cols * (int64_t)ctx->M), NETMAX_STATIC_MAX_VALUES);
  if (n_cols == 0) return NETMAX_OK;
  for (int64_t k = 0; k < n_cols; ++k)
    if (host_cols[k] < 0 || host_cols[k] >= ctx->d) return fail(ctx, NETMAX_INVALID_ARG, "cols[%lld] = %lld outside [0, d)", (long long)k, (long long)host_cols[k]);
  DeviceGuard guard(ctx->device);
  StaticGatherScratch* scratch = nullptr;
  int rc = gather_scratch_address(ctx, &scratch);
  if (rc) return rc;
  const int64_t total = n_cols * ctx->M;
  const int grid = (int)std::min<int64_t>((total + kThreads - 1) / kThreads, 4096);
  NM_CUDA(ctx, cudaMemcpyAsync(scratch->cols, host_cols, (size_t)n_cols * sizeof(int64_t), cudaMemcpyHostToDevice, ctx->stream));
  gather_columns_kernel<<<grid, kThreads, 0, ctx->stream>>>(ctx->x[ctx->cur], ctx->storage == NETMAX_STORAGE_BF16, ctx->L.ld, ctx->M, scratch->cols, n_cols, scratch->values);
  ctx->launches += 1;
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(host_out, scratch->values, (size_t)total * sizeof(float), cudaMemcpyDeviceToHost, ctx->stream);
  // whatever happened, leave the shared array idle: the next call, perhaps on another stream, reuses it
  const int rs = synchronise(ctx);
  if (e != cudaSuccess) return fail(ctx, NETMAX_CUDA_ERROR, "read_columns_static: %s", cudaGetErrorString(e));
  return rs;
}

static int ring_range(netmax_ctx* ctx, int64_t first, int64_t n) {
  if (first < ctx->round0 || n < 0 || first + n > ctx->rounds || first < ctx->rounds - ctx->trace_rounds)
    return fail(ctx, NETMAX_TRACE_RANGE, "rounds [%lld, %lld) are not in the ring (rounds done %lld, capacity %lld)",
                (long long)first, (long long)(first + n), (long long)ctx->rounds, (long long)ctx->trace_rounds);
  return NETMAX_OK;
}

int netmax_peer_trace(netmax_ctx* ctx, int64_t first_round, int64_t n, int32_t* host_out) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  int rc = ring_range(ctx, first_round, n);
  if (rc) return rc;
  if (n == 0) return NETMAX_OK;
  if (!host_out) return fail(ctx, NETMAX_INVALID_ARG, "host_out is NULL");
  DeviceGuard guard(ctx->device);
  ctx->trace_read = true;
  bool mirrored = ctx->trace_mirror != nullptr;
  for (int64_t r = first_round; mirrored && r < first_round + n; ++r) mirrored = (ctx->on_host[(size_t)(r % ctx->trace_rounds)] & 2) != 0;
  if (mirrored) {
    rc = synchronise(ctx);
    if (rc) return rc;
  }
  const size_t row = (size_t)ctx->M * sizeof(int32_t);
  int64_t r = first_round;
  while (r < first_round + n) {  // at most two contiguous pieces of the ring
    const int64_t slot = r % ctx->trace_rounds;
    const int64_t piece = std::min<int64_t>(first_round + n - r, ctx->trace_rounds - slot);
    int32_t* out = host_out + (size_t)(r - first_round) * ctx->M;
    if (mirrored) std::memcpy(out, ctx->trace_mirror + (size_t)slot * ctx->M, piece * row);
    else if ((rc = read_back(ctx, out, ctx->trace + (size_t)slot * ctx->M, piece * row)) != NETMAX_OK) return rc;
    r += piece;
  }
  return NETMAX_OK;
}

int netmax_telemetry(netmax_ctx* ctx, int64_t first_round, int64_t n, double* host_consensus, double* host_loss) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  int rc = ring_range(ctx, first_round, n);
  if (rc) return rc;
  if (n == 0) return NETMAX_OK;
  DeviceGuard guard(ctx->device);
  ctx->tel_read = true;
  auto in_host = [&](int64_t slot) { return ctx->tel_host && (ctx->on_host[(size_t)slot] & 1); };
  bool all = true;
  for (int64_t k = 0; all && k < n; ++k) all = in_host((first_round + k) % ctx->trace_rounds);
  std::vector<double> copy;
  if (all) {
    rc = synchronise(ctx);
  } else {
    copy.resize((size_t)ctx->trace_rounds * 2);
    rc = read_back(ctx, copy.data(), ctx->tel_dev, copy.size() * sizeof(double));
  }
  if (rc) return rc;
  for (int64_t k = 0; k < n; ++k) {
    const int64_t slot = (first_round + k) % ctx->trace_rounds;
    const double* ring = in_host(slot) ? ctx->tel_host : copy.data();
    if (host_consensus) host_consensus[k] = ring[2 * slot];
    if (host_loss) host_loss[k] = ring[2 * slot + 1];
  }
  return NETMAX_OK;
} NM_CATCH_CTX(ctx)

int netmax_replicas_device(netmax_ctx* ctx, const float** x, int64_t* ld) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!x || !ld) return fail(ctx, NETMAX_INVALID_ARG, "output pointer is NULL");
  ctx->replicas_exposed = true;  // (the caller may write through the address: what was mirrored may be stale from now on)
  ctx->staged = false;
  *x = reinterpret_cast<const float*>(ctx->x[ctx->cur]);
  *ld = ctx->L.ld;
  return NETMAX_OK;
}

int netmax_sample_peers(netmax_ctx* ctx, int64_t first_round, int64_t n_rounds, int32_t* device_out) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (first_round < 0 || n_rounds < 0 || (n_rounds > 0 && !device_out)) return fail(ctx, NETMAX_INVALID_ARG, "bad range or NULL output");
  DeviceGuard guard(ctx->device);
  return launch_sampler(ctx, (uint64_t)first_round, n_rounds, device_out, nullptr, 0, INT64_MAX);
} NM_CATCH_CTX(ctx)

// ---- telemetry on demand --------------------------------------------------------------------
int netmax_measure(netmax_ctx* ctx, double* consensus, double* loss) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  DeviceGuard guard(ctx->device);
  RoundPlan plan;
  int rc = plan_round(ctx, plan, 2);  // 2: the measuring instantiation of the round kernel
  if (rc) return rc;
  RoundKernel kernel = pick_kernel(2, plan.short_vectors, ctx->L.halves);
  RoundParams p;
  std::memset(&p, 0, sizeof p);
  p.x_cur = reinterpret_cast<const float4*>(ctx->x[ctx->cur]);
  p.x_nxt = nullptr;
  p.c = reinterpret_cast<const float4*>(ctx->c);
  p.peers = nullptr;
  p.wtab = ctx->wtab;
  p.partials = ctx->partials;
  p.ticket = ctx->ticket;
  p.tel_out = ctx->measure_out;
  p.ldq = ctx->L.ldq;
  p.row_bytes = (uint32_t)(ctx->L.ld * ctx->L.elem);
  p.nq = ctx->L.nq;
  p.n_tiles = plan.n_tiles;
  p.M = ctx->M;
  p.tail = (int32_t)(ctx->d % (4 * ctx->L.halves));
  p.cg = plan.cg;
  p.rl = plan.rl;
  p.rg = plan.rg;
  p.rows_per_group = plan.rows_per_group;
  p.colpart = ctx->colpart;
  p.coltick = ctx->coltick;
  p.inv_M = 1.0f / (float)ctx->M;
  p.keys = ctx->keys;
  ctx->host_writes = true;
  kernel<<<plan.grid, kThreads, plan.smem, ctx->stream>>>(p);
  ctx->launches += 1;
  NM_CUDA(ctx, cudaGetLastError());
  rc = synchronise(ctx);
  if (consensus) *consensus = ctx->measure_out[0];
  if (loss) *loss = ctx->measure_out[1];
  return rc;
}

// ---- asynchronous timeline --------------------------------------------------------------------
// First word of the Philox block of the peer stream at counter (0, worker, iteration): the host
// twin of the device sampler (same published algorithm, 32x32->64 products and xors).
static uint32_t host_peer_word(const PhiloxKeys& keys, uint32_t worker, uint64_t iter) {
  uint32_t c0 = 0, c1 = worker, c2 = (uint32_t)iter, c3 = philox_ctr3(kTagPeer, iter);
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)kPhiloxMul0 * c0, p1 = (uint64_t)kPhiloxMul1 * c2;
    const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ keys.k0[r];
    const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ keys.k1[r];
    c0 = n0;
    c1 = (uint32_t)p1;
    c2 = n2;
    c3 = (uint32_t)p0;
  }
  return c0;
}

// Draws the peer of worker i's next local iteration (Algorithm 2) and sets when it will finish.
// The policy is read at the top of an iteration and the moving average records the time the
// iteration took, so the pull weight and the duration are latched here: a policy or time
// matrix that arrives while the iteration is in flight does not touch them.
static void async_start_iteration(netmax_ctx* ctx, int i, double start) {
  const int32_t M = ctx->M;
  const uint32_t u = host_peer_word(ctx->keys, (uint32_t)i, (uint64_t)ctx->local_n[i]);
  const uint32_t* row = ctx->h_thr.data() + (size_t)i * M;
  const int32_t count = (int32_t)(std::upper_bound(row, row + M, u) - row);  // #{j : T[j] <= u}
  const int32_t m = std::min(count, ctx->h_last[i]);
  const size_t link = (size_t)i * M + m;
  ctx->pending_peer[i] = m;
  ctx->pending_weight[i] = (m == i) ? 0.0f : ctx->h_w[link];
  ctx->pending_duration[i] = ctx->t_iter[link];
  ctx->finish[i] = start + ctx->pending_duration[i];
}

int netmax_async_begin(netmax_ctx* ctx, const double* t_iter, double beta) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (ctx->rounds != ctx->round0) return fail(ctx, NETMAX_INVALID_ARG, "netmax_async_begin must precede any netmax_round");
  if (!(beta >= 0.0 && beta < 1.0)) return fail(ctx, NETMAX_INVALID_ARG, "beta = %g outside [0, 1)", beta);
  const int32_t M = ctx->M;
  if (t_iter) {
    for (size_t k = 0; k < (size_t)M * M; ++k) {
      const int i = (int)(k / M), m = (int)(k % M);
      const bool used = (i == m) || ctx->adj[k];
      if (used && !(t_iter[k] > 0.0 && std::isfinite(t_iter[k])))
        return fail(ctx, NETMAX_INVALID_ARG, "t_iter[%d,%d] = %g must be positive and finite", i, m, t_iter[k]);
    }
    ctx->t_iter.assign(t_iter, t_iter + (size_t)M * M);
  }
  {
    DeviceGuard guard(ctx->device);
    int rc = need_host_tables(ctx);
    if (rc) return rc;
  }
  ctx->async_on = false;  // until all of the state below is there
  ctx->beta = beta;
  ctx->now = 0.0;
  ctx->steps = 0;
  ctx->local_n.assign(M, 0);
  ctx->pending_peer.assign(M, 0);
  ctx->pending_weight.assign(M, 0.0f);
  ctx->pending_duration.assign(M, 0.0);
  ctx->finish.assign(M, 0.0);
  ctx->ema.assign((size_t)M * M, 0.0);
  ctx->ema_count.assign((size_t)M * M, 0);
  ctx->ev_cap = std::max<int64_t>(ctx->trace_rounds * (int64_t)M, 1024);
  ctx->ev_worker.assign(ctx->ev_cap, 0);
  ctx->ev_peer.assign(ctx->ev_cap, 0);
  ctx->ev_n.assign(ctx->ev_cap, 0);
  ctx->ev_time.assign(ctx->ev_cap, 0.0);
  ctx->step_writes.assign(M, 0);
  ctx->step_reads.assign(M, 0);
  ctx->queue.clear();
  for (int i = 0; i < M; ++i) {
    async_start_iteration(ctx, i, 0.0);
    ctx->queue.emplace_back(ctx->finish[i], i);
  }
  std::make_heap(ctx->queue.begin(), ctx->queue.end(), std::greater<std::pair<double, int>>());
  ctx->async_on = true;
  return NETMAX_OK;
} NM_CATCH_CTX(ctx)

int netmax_async_set_times(netmax_ctx* ctx, const double* t_iter) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!t_iter) return fail(ctx, NETMAX_INVALID_ARG, "t_iter is NULL");
  ctx->t_iter.assign(t_iter, t_iter + (size_t)ctx->M * ctx->M);
  return NETMAX_OK;
} NM_CATCH_CTX(ctx)

// Network Monitor (Algorithm 1): collect the workers' moving averages of iteration times, run
// Algorithm 3 on them and send P and rho back.  An average that has seen n samples is read as
// T / (1 - beta^n) (Algorithm 2 starts T at 0); a link that was never sampled is taken at its
// current iteration time.  An infeasible grid leaves the policy in force.
static int monitor_refresh(netmax_ctx* ctx) {
  const int32_t M = ctx->M;
  std::vector<double> t((size_t)M * M, 0.0);
  for (size_t at = 0; at < (size_t)M * M; ++at) {
    const int i = (int)(at / M), m = (int)(at % M);
    if (i != m && !ctx->adj[at]) continue;
    const int64_t n = ctx->ema_count[at];
    t[at] = n > 0 ? ctx->ema[at] / (1.0 - std::pow(ctx->beta, (double)n)) : ctx->t_iter[at];
  }
  std::vector<double> P((size_t)M * M);
  double rho = 0.0;
  const bool fixed = ctx->pull_weight > 0.0;  // constant pull weight: the extension section's form of Algorithm 3
  double floor_sel = 0.0;
  int rc = fixed ? netmax_policy_generate_fixed_weight(M, t.data(), ctx->adj.data(), ctx->pull_weight, ctx->policy_K, ctx->policy_R,
                                                       ctx->policy_rho_upper, P.data(), &floor_sel, nullptr)
                 : generate_policy(ctx, t.data(), P.data(), &rho);
  if (rc == NETMAX_INFEASIBLE) return NETMAX_OK;
  if (rc) return fail(ctx, rc, "%s", netmax_last_error(nullptr));
  ctx->P.swap(P);
  if (!fixed) ctx->rho = rho;
  ctx->monitor_refreshes += 1;
  rc = upload_policy(ctx);
  return rc ? rc : need_host_tables(ctx);
}

int netmax_async_monitor(netmax_ctx* ctx, double period_s) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!ctx->async_on) return fail(ctx, NETMAX_INVALID_ARG, "call netmax_async_begin first");
  if (!(period_s >= 0.0) || !std::isfinite(period_s)) return fail(ctx, NETMAX_INVALID_ARG, "period_s = %g", period_s);
  ctx->monitor_period = period_s;
  ctx->monitor_next = ctx->now + period_s;
  return NETMAX_OK;
}

int64_t netmax_async_monitor_refreshes(const netmax_ctx* ctx) { return ctx ? ctx->monitor_refreshes : -1; }

// Replaces the smallest entry of a binary heap (one way down instead of a pop and a push).
static void replace_top(std::vector<std::pair<double, int>>& heap, std::pair<double, int> entry) {
  const size_t n = heap.size();
  size_t at = 0;
  for (;;) {
    size_t child = 2 * at + 1;
    if (child >= n) break;
    if (child + 1 < n && heap[child + 1] < heap[child]) ++child;
    if (!(heap[child] < entry)) break;
    heap[at] = heap[child];
    at = child;
  }
  heap[at] = entry;
}

constexpr int64_t kEventsAhead = 4 * kStepTileEvents;

// Consecutive global steps, one launch for as many as touch disjoint replicas.  *used: how many were enqueued -- with
// more events to come (!last) a launch that could still take some waits for them.
static int enqueue_disjoint_steps(netmax_ctx* ctx, const StepEvent* events, int64_t n, bool last, int64_t* used) {
  StepKernel kernel = pick_step_kernel(ctx->objective, ctx->L.halves);
  StepParams p;
  p.x = reinterpret_cast<float4*>(ctx->x[ctx->cur]);
  p.c = reinterpret_cast<const float4*>(ctx->c);
  p.nq = ctx->L.nq;
  p.row_bytes = (uint32_t)(ctx->L.ld * ctx->L.elem);
  p.tail = (int32_t)(ctx->d % (4 * ctx->L.halves));
  p.alpha = (float)ctx->alpha;
  p.sigma = noise_scale(ctx);
  p.q_offset = ctx->q_offset;
  p.keys = ctx->keys;
  uint8_t *const writes = ctx->step_writes.data(), *const reads = ctx->step_reads.data();
  *used = 0;
  for (int64_t done = 0; done < n;) {
    p.n_events = 0;
    // a step must not write a row that an earlier step of the launch reads or writes, nor read a row that one writes
    while (done < n && p.n_events < kMaxStepEvents) {
      const StepEvent& e = events[done];
      if (writes[e.worker] || reads[e.worker] || writes[e.peer]) break;
      writes[e.worker] = reads[e.worker] = reads[e.peer] = 1;
      p.ev[p.n_events++] = e;
      ++done;
    }
    for (int e = 0; e < p.n_events; ++e) writes[p.ev[e].worker] = reads[p.ev[e].worker] = reads[p.ev[e].peer] = 0;
    if (!last && done == n && p.n_events < kMaxStepEvents) break;
    *used = done;
    const int64_t want = (ctx->L.nq + kThreads - 1) / kThreads;
    const int64_t cap = std::max<int64_t>(1, (int64_t)8 * ctx->sm_count / p.n_events);
    dim3 grid((unsigned)std::min<int64_t>(want, cap), (unsigned)p.n_events);
    kernel<<<grid, kThreads, 0, ctx->stream>>>(p);
    ctx->launches += 1;
  }
  NM_CUDA(ctx, cudaGetLastError());
  return NETMAX_OK;
}

using StepTileKernel = void (*)(const StepTileParams);
static StepTileKernel pick_step_tile_kernel(int objective, int halves) {
  if (halves == 2) return objective == 1 ? step_tiles_kernel<1, true> : step_tiles_kernel<0, true>;
  return objective == 1 ? step_tiles_kernel<1, false> : step_tiles_kernel<0, false>;
}

// Launch shape of step_tiles_kernel, and whether it pays: microseconds of a step in either kernel and of bringing the
// columns on chip.  A thread takes 32 M bytes of shared memory.  Measured: a step of a column group takes a scheduler
// 172 cycles with warps enough (8 workers: 12.8 us per step of 11.2 M elements against 27.1) and 480 with a single one
// (32 workers, 1.5 warps: 4.3 us of 2 M elements against 5.2; 36 workers, one warp: 6.4 by this rule, not taken);
// step_kernel moves 16 bytes per element at 6.2 TB/s, but a step takes half a microsecond of launches at least.
struct StepTilePlan {
  int threads = 0;
  int64_t per_sm = 0;
  double tile_us = 0, step_us = 0, load_us = 0;
  bool pays(int64_t steps) const {  // (every launch brings the rows in)
    const int64_t launches = (steps + kStepTileEvents - 1) / kStepTileEvents;
    return threads > 0 && (double)steps * (step_us - tile_us) > (double)launches * load_us;
  }
};
static StepTilePlan plan_step_tiles(const netmax_ctx* ctx) {
  StepTilePlan f;
  const int64_t M = ctx->M, nq = (ctx->d + 3) / 4;
  const size_t head = step_tile_head(kStepTileEvents, M);
  int64_t best_warps = 0;
  for (int threads : {256, 128, 64, 32}) {
    const size_t smem = head + (size_t)32 * M * threads;
    if (smem > (size_t)226 * 1024) continue;
    const int64_t fit = std::min<int64_t>(512 / threads, (int64_t)((size_t)228 * 1024 / (smem + 1024)));
    // no more warps than the column groups fill; narrow CTAs only where they bring more of them (fewer than four warps
    // do not spread over the four schedulers by themselves), or where everything is resident in them
    const int64_t warps = std::min<int64_t>(fit * threads / 32, std::max<int64_t>(1, (nq / 32 + ctx->sm_count - 1) / ctx->sm_count));
    const bool spread = threads == 32 && (nq + 31) / 32 <= fit * ctx->sm_count;
    if (warps > best_warps || (spread && warps >= best_warps)) {
      best_warps = warps;
      f.threads = threads;
      f.per_sm = fit;
    }
  }
  if (f.threads == 0) return f;
  const double items = (double)nq / 32.0 / (4.0 * ctx->sm_count), bytes = (double)ctx->d * ctx->L.elem;
  f.tile_us = std::max(1.0, items) * std::max(172.0, 480.0 / std::min(1.0 * std::max(1.0, best_warps / 4.0), std::max(1.0, items))) / 1965.0;
  if (best_warps < 4 && items > 1.0) f.tile_us *= 4.0 / (double)best_warps;  // (schedulers without a warp)
  // Narrow CTAs, one or two to an SM (many workers): every lap is a thread's chain of steps, and its rows come in one after
  // the other, four bfloat16 ones at a time (100 workers, 64 steps of 41,946 elements in two laps: 77 us in bfloat16 and 42
  // in fp32 against 33 in launches of disjoint steps; 64 workers, 16 steps of 4,099: 20 against 13).
  const double laps = std::ceil((double)((nq + f.threads - 1) / f.threads) / (double)(f.per_sm * ctx->sm_count));
  f.tile_us = std::max(f.tile_us, laps * 480.0 / 1965.0 * (best_warps <= 4 ? 1.0 : 4.0 / (double)best_warps));
  f.step_us = std::max(0.5, 4.0 * bytes / 6.2e6);
  // (12 M bytes, a quarter of it beside the steps; or the rows' latencies)
  f.load_us = 3.0 + std::max(2.2 * (double)M * bytes / 6.2e6, laps * (double)M * (ctx->L.halves == 2 ? 0.25 : 0.08));
  return f;
}

// Enqueues the collected events and takes them out of the list (see enqueue_disjoint_steps).
static int enqueue_steps(netmax_ctx* ctx, std::vector<StepEvent>& events, const StepTilePlan& plan, bool last) {
  const int64_t n = (int64_t)events.size();
  const int threads = plan.threads;
  int64_t done = 0;
  if (plan.pays(n)) {
    StepTileKernel kernel = pick_step_tile_kernel(ctx->objective, ctx->L.halves);
    StepTileParams p;
    p.x = reinterpret_cast<char*>(ctx->x[ctx->cur]);
    p.c = reinterpret_cast<const char*>(ctx->c);
    p.nq = (ctx->d + 3) / 4;
    p.n_tiles = (p.nq + threads - 1) / threads;
    p.row_bytes = (uint32_t)(ctx->L.ld * ctx->L.elem);
    p.M = ctx->M;
    p.tail = (int32_t)(ctx->d % 4);
    p.alpha = (float)ctx->alpha;
    p.sigma = noise_scale(ctx);
    p.q_offset = ctx->q_offset;
    p.keys = ctx->keys;
    const size_t slabs = (size_t)32 * ctx->M * threads;
    NM_CUDA(ctx, allow_smem((const void*)kernel, step_tile_head(kStepTileEvents, ctx->M) + slabs));
    const unsigned grid = (unsigned)std::min<int64_t>(p.n_tiles, plan.per_sm * ctx->sm_count);
    while (done < n) {
      const int64_t launches_left = (n - done + kStepTileEvents - 1) / kStepTileEvents;  // launches of even length
      p.n_events = (int32_t)((n - done + launches_left - 1) / launches_left);
      for (int e = 1; e < p.n_events; ++e)  // one high word of the iteration per launch
        if (events[done + e].ctr3 != events[done].ctr3) p.n_events = e;
      std::memcpy(p.ev, events.data() + done, p.n_events * sizeof(StepEvent));
      kernel<<<grid, threads, step_tile_head(p.n_events, ctx->M) + slabs, ctx->stream>>>(p);
      ctx->launches += 1;
      done += p.n_events;
    }
    NM_CUDA(ctx, cudaGetLastError());
  }
  int64_t used = 0;
  const int rc = enqueue_disjoint_steps(ctx, events.data() + done, n - done, last, &used);
  events.erase(events.begin(), events.begin() + done + used);
  return rc;
}

int netmax_async_steps(netmax_ctx* ctx, int64_t n_steps) try {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!ctx->async_on) return fail(ctx, NETMAX_INVALID_ARG, "call netmax_async_begin first");
  ctx->staged = false;
  if (n_steps < 0) return fail(ctx, NETMAX_INVALID_ARG, "n_steps = %lld < 0", (long long)n_steps);
  DeviceGuard guard(ctx->device);
  const int32_t M = ctx->M;
  // Events are collected and enqueued some hundred at a time: the GPU runs them while the clocks go on.
  std::vector<StepEvent> events;
  events.reserve((size_t)std::min<int64_t>(n_steps, kEventsAhead));
  const StepTilePlan plan = plan_step_tiles(ctx);
  // (events of single launches go out soon: the host's part is the longer one there)
  const size_t ahead = plan.pays(kEventsAhead) ? (size_t)kEventsAhead : 8;
  size_t due = ahead;
  int64_t ev_slot = ctx->steps % ctx->ev_cap;
  auto flush = [&](bool last) {
    const int rc = enqueue_steps(ctx, events, plan, last);
    due = events.size() + ahead;
    return rc;
  };
  for (int64_t k = 0; k < n_steps; ++k) {
    // the next global step: the worker whose iteration finishes first (ties: lowest index)
    const int i = ctx->queue[0].second;
    // the Network Monitor wakes up before any step at or after its next period boundary
    while (ctx->monitor_period > 0.0 && ctx->finish[i] >= ctx->monitor_next) {
      int rc = flush(true);
      if (!rc) rc = monitor_refresh(ctx);
      if (rc) return rc;
      ctx->monitor_next += ctx->monitor_period;
    }
    const int m = ctx->pending_peer[i];
    if (events.size() >= due) {
      int rc = flush(false);
      if (rc) return rc;
    }
    const uint64_t n = (uint64_t)ctx->local_n[i];
    events.push_back(StepEvent{i, m, (uint32_t)n, philox_ctr3(kTagNoise, n), ctx->pending_weight[i]});
    // bookkeeping of Algorithm 2: the clock, the EMA of the iteration time, the next iteration
    ctx->now = ctx->finish[i];
    const int64_t slot = ev_slot;
    ev_slot = ev_slot + 1 == ctx->ev_cap ? 0 : ev_slot + 1;
    ctx->ev_worker[slot] = i;
    ctx->ev_peer[slot] = m;
    ctx->ev_n[slot] = (int64_t)n;
    ctx->ev_time[slot] = ctx->now;
    const size_t at = (size_t)i * M + m;
    ctx->ema[at] = ctx->beta * ctx->ema[at] + (1.0 - ctx->beta) * ctx->pending_duration[i];
    ctx->ema_count[at] += 1;
    ctx->local_n[i] += 1;
    ctx->steps += 1;
    async_start_iteration(ctx, i, ctx->now);
    replace_top(ctx->queue, {ctx->finish[i], i});
  }
  return flush(true);
} NM_CATCH_CTX(ctx)

int netmax_async_time(netmax_ctx* ctx, double* sim_time, int64_t* steps_done) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!ctx->async_on) return fail(ctx, NETMAX_INVALID_ARG, "call netmax_async_begin first");
  if (sim_time) *sim_time = ctx->now;
  if (steps_done) *steps_done = ctx->steps;
  return NETMAX_OK;
}

int netmax_async_trace(netmax_ctx* ctx, int64_t first_step, int64_t n, int32_t* worker, int32_t* peer, int64_t* local_iter,
                       double* finish_time) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!ctx->async_on) return fail(ctx, NETMAX_INVALID_ARG, "call netmax_async_begin first");
  if (first_step < 0 || n < 0 || first_step + n > ctx->steps || first_step < ctx->steps - ctx->ev_cap)
    return fail(ctx, NETMAX_TRACE_RANGE, "steps [%lld, %lld) are not in the ring (steps done %lld, capacity %lld)",
                (long long)first_step, (long long)(first_step + n), (long long)ctx->steps, (long long)ctx->ev_cap);
  for (int64_t k = 0; k < n; ++k) {
    const int64_t slot = (first_step + k) % ctx->ev_cap;
    if (worker) worker[k] = ctx->ev_worker[slot];
    if (peer) peer[k] = ctx->ev_peer[slot];
    if (local_iter) local_iter[k] = ctx->ev_n[slot];
    if (finish_time) finish_time[k] = ctx->ev_time[slot];
  }
  return NETMAX_OK;
}

int netmax_async_ema(netmax_ctx* ctx, double* ema_out, int64_t* samples_out) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (!ctx->async_on) return fail(ctx, NETMAX_INVALID_ARG, "call netmax_async_begin first");
  if (ema_out) std::memcpy(ema_out, ctx->ema.data(), ctx->ema.size() * sizeof(double));
  if (samples_out) std::memcpy(samples_out, ctx->ema_count.data(), ctx->ema_count.size() * sizeof(int64_t));
  return NETMAX_OK;
}

int netmax_launch_shape(netmax_ctx* ctx, int64_t n_rounds, netmax_shape* out) try {
  if (!ctx || !out) return fail(ctx, NETMAX_INVALID_ARG, "ctx or out is NULL");
  if (n_rounds < 1) return fail(ctx, NETMAX_INVALID_ARG, "n_rounds = %lld < 1", (long long)n_rounds);
  DeviceGuard guard(ctx->device);
  RoundPlan plan;
  PipePlan pipe;
  FusedPlan fused;
  TilePlan tiles;
  int rc = plan_round(ctx, plan, ctx->objective);
  if (!rc) rc = plan_call(ctx, plan, pipe, fused, tiles);
  if (rc) return rc;
  std::memset(out, 0, sizeof *out);
  out->kernel = batch_kernel(ctx, plan, pipe, fused, tiles, std::min(n_rounds, ctx->trace_rounds));
  switch (out->kernel) {
    case NETMAX_KERNEL_PIPE:
      out->groups = pipe.G;
      out->rows = pipe.rows;
      out->warps = pipe.movers + pipe.helpers;
      break;
    case NETMAX_KERNEL_TILES:
      out->groups = tiles.G;
      out->rows = tiles.rows;
      out->warps = tiles.threads / 32;
      out->own_instance = ctx->objective == 1 && tile_shape_of_its_own(tiles.rows, tiles.G, tiles.threads / 32);
      break;
    case NETMAX_KERNEL_FUSED:
      out->groups = fused.threads;
      out->rows = ctx->M;
      out->warps = fused.threads / 32;
      break;
    default:
      out->groups = plan.cg;
      out->rows = (int32_t)((plan.rows_per_group + plan.rl - 1) / plan.rl);
      out->warps = kThreads / 32;
  }
  return NETMAX_OK;
} NM_CATCH_CTX(ctx)

int netmax_debug_absent_ctas(netmax_ctx* ctx, int32_t n) {
  if (!ctx) return fail(nullptr, NETMAX_INVALID_ARG, "ctx is NULL");
  if (n < 0 || n > 1024) return fail(ctx, NETMAX_INVALID_ARG, "n = %d outside [0, 1024]", n);
  ctx->inject_absent_ctas = (uint32_t)n;
  return NETMAX_OK;
}

int64_t netmax_kernel_launches(const netmax_ctx* ctx) { return ctx ? ctx->launches : -1; }

const char* netmax_last_error(const netmax_ctx* ctx) { return ctx ? ctx->error.c_str() : g_error.c_str(); }

}  // extern "C"
