// Communication-policy generation (Algorithm 3) on the GPU, for large M.
//
// Same readings and the same per-row solution as the host generator (netmax_policy.cpp): the
// grids rho_k = k U_rho / K and t_bar_r = U - (R - r)(U - L)/R; per grid point the row-wise LP
// optimum (Eq. 14 under Eq. 10-13: floor + exponential tilt, or least p_ii + fastest peers),
// Y_P (Eq. 22 with p_i = 1/M), its second largest eigenvalue by Lanczos on the complement of
// the all-ones vector, and the arg-min of t_bar ln(eps) / ln(lambda_2).  One CTA solves one row;
// the M x M matrices t, P and Y stay in device memory in fp64.
#include "../../include/netmax.h"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

#include "netmax_fp64.cuh"
#include "netmax_policy.h"

namespace {

using netmax::exp_table;
using netmax::fast_reciprocal;
using netmax::kExpTable;
using netmax::table_exp;

constexpr int kRowThreads = 256;
constexpr double kEtaCap = 600.0;
constexpr double kTie = 1e-12;
constexpr double kEps = 1e-3;

struct RowInfo {  // per row, independent of the grid point
  double C, tmin, tmax, sum_f1, sum_f1t;
  double mean_lo, mean_hi;  // mean of the times mapped to [0, 1] at the ends of the bracket, eta = -+kEtaCap
  int n_nb, n_fast;
  int both;                 // every link of the row is there in both directions: d_im + d_mi = 2
};

__device__ __forceinline__ double warp_sum(double v) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  return v;
}

// Sum of v over the CTA, returned to every thread.  s_buf: 33 doubles.
__device__ double block_sum(double v, double* s_buf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) s_buf[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double t = lane < nw ? s_buf[lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) s_buf[32] = t;
  }
  __syncthreads();
  return s_buf[32];
}

__device__ double block_min(double v, double* s_buf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int off = 16; off > 0; off >>= 1) v = fmin(v, __shfl_down_sync(0xffffffffu, v, off));
  __syncthreads();
  if (lane == 0) s_buf[warp] = v;
  __syncthreads();
  if (warp == 0) {
    double t = lane < nw ? s_buf[lane] : INFINITY;
    for (int off = 16; off > 0; off >>= 1) t = fmin(t, __shfl_down_sync(0xffffffffu, t, off));
    if (lane == 0) s_buf[32] = t;
  }
  __syncthreads();
  return s_buf[32];
}

__global__ void __launch_bounds__(kRowThreads) row_info_kernel(int M, const double* t, const uint8_t* adj, RowInfo* info) {
  __shared__ double s_buf[33];
  const int i = blockIdx.x;
  double f1s = 0, f1t = 0, mn = INFINITY, mx = -INFINITY, nb = 0, one_way = 0;
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    if (m == i || !adj[(size_t)i * M + m]) continue;
    const double tm = t[(size_t)i * M + m];
    const double f1 = (double)adj[(size_t)i * M + m] + (double)adj[(size_t)m * M + i];
    f1s += f1;
    f1t += f1 * tm;
    one_way += f1 != 2.0;
    mn = fmin(mn, tm);
    mx = fmax(mx, tm);
    nb += 1;
  }
  f1s = block_sum(f1s, s_buf);
  f1t = block_sum(f1t, s_buf);
  nb = block_sum(nb, s_buf);
  mn = block_min(mn, s_buf);
  mx = -block_min(-mx, s_buf);
  double fast = 0;
  for (int m = threadIdx.x; m < M; m += blockDim.x)
    if (m != i && adj[(size_t)i * M + m] && t[(size_t)i * M + m] <= mn * (1.0 + kTie)) fast += 1;
  fast = block_sum(fast, s_buf);
  one_way = block_sum(one_way, s_buf);
  double mean[2] = {0.0, 0.0};
  const double scale = mx - mn;
  if (scale > kTie * mx) {
    for (int e = 0; e < 2; ++e) {
      const double eta = e == 0 ? -kEtaCap : kEtaCap;
      double a0 = 0, a1 = 0;
      for (int m = threadIdx.x; m < M; m += blockDim.x) {
        if (m == i || !adj[(size_t)i * M + m]) continue;
        const double sv = (t[(size_t)i * M + m] - mn) / scale, w = exp(-eta * sv);
        a0 += w;
        a1 += w * sv;
      }
      a0 = block_sum(a0, s_buf);
      a1 = block_sum(a1, s_buf);
      mean[e] = a1 / a0;
    }
  }
  if (threadIdx.x == 0) {
    RowInfo r;
    r.mean_lo = mean[0];
    r.mean_hi = mean[1];
    r.both = one_way == 0.0;
    r.C = t[(size_t)i * M + i];
    r.tmin = mn;
    r.tmax = mx;
    r.sum_f1 = f1s;
    r.sum_f1t = f1t;
    r.n_nb = (int)nb;
    r.n_fast = (int)fast;
    info[i] = r;
  }
}

// Sums of three or four values over the CTA, returned to every thread.  s_buf: 33 doubles for each.
template <int kValues>
__device__ void block_sums(double (&v)[kValues], double* s_buf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < kValues; ++k) v[k] = warp_sum(v[k]);
  __syncthreads();
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < kValues; ++k) s_buf[33 * k + warp] = v[k];
  }
  __syncthreads();
  if (warp < kValues) {
    double t = lane < nw ? s_buf[33 * warp + lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) s_buf[33 * warp + 32] = t;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kValues; ++k) v[k] = s_buf[33 * k + 32];
}
__device__ __forceinline__ void block_sum3(double& a, double& b, double& c, double* s_buf) {
  double v[3] = {a, b, c};
  block_sums(v, s_buf);
  a = v[0];
  b = v[1];
  c = v[2];
}
__device__ __forceinline__ void block_sum4(double& a, double& b, double& c, double& d, double* s_buf) {
  double v[4] = {a, b, c, d};
  block_sums(v, s_buf);
  a = v[0];
  b = v[1];
  c = v[2];
  d = v[3];
}

// Grid points t_bar_r, r = first + 1 ... first + n, of one rho: alpha rho and the inner grid.
struct PointGrid {
  double ar, U, delta;
  int R, first, n;
  // T = M t_bar_r, t_bar_r = U - (R - r) delta, one rounding per operation as on the host
  __device__ __forceinline__ double time(int M, int k) const { return __dmul_rn((double)M, __dsub_rn(U, __dmul_rn((double)(R - 1 - first - k), delta))); }
};
// A row of the LP at one grid point: p_im = alpha rho (d_im + d_mi) + share exp(-eta s_m), or, with p_ii > 0 or equal
// times (eta unused), the share on the fastest links or on all.
enum RowKind : int { kNoRow = 0, kTilted, kEven, kFastest };
struct RowPoint {
  double eta, share, pii;
  int kind;
};
// Where a row's search stands: eta of the last point solved, and mean, variance and third central moment of s under its
// weights (var = 0: none yet).
struct RowState {
  double eta, mean, var, third;
};

// One row of the LP at the points of a grid; a row without a solution is kNoRow and raises infeasible[point].  Bound by fp64
// exponentials: the row's times, mapped to [0, 1], stay in shared memory (-1: no link) for all points and steps.  The steps are
// Halley's: the mean's first two derivatives are moments that come with it (d mean / d eta = -var, d var / d eta = -third).
// They start from the previous point's solution, whose moments are known, so that the first step costs nothing; two or three
// passes over the row follow.  4,096 workers, eight grid points per launch: 1,085 us with Newton's steps from a pass at the old
// solution on and the library's exp, 725 so; with a launch per grid point, which reads the times every time and stores P, 171 us
// per point.
__global__ void __launch_bounds__(kRowThreads) row_solve_kernel(int M, const double* t, const uint8_t* adj, const RowInfo* info,
                                                                const PointGrid grid, RowState* state, RowPoint* points, int* infeasible) {
  extern __shared__ double s_time[];
  __shared__ double s_buf[132], s_table[kExpTable];
  const int i = blockIdx.x;
  const RowInfo r = info[i];
  const double* ti = t + (size_t)i * M;
  const uint8_t* ai = adj + (size_t)i * M;
  const double F = grid.ar * r.sum_f1;
  const double free_mass = 1.0 - F, A = grid.ar * r.sum_f1t;
  const double lo = A + free_mass * r.tmin, hi = A + free_mass * r.tmax;
  const double scale = r.tmax - r.tmin;
  const bool flat = !(scale > kTie * r.tmax) || free_mass <= 0.0;
  if (!flat) {
    const double inv_scale = 1.0 / scale;
    for (int m = threadIdx.x; m < M; m += blockDim.x) s_time[m] = (m != i && ai[m]) ? (ti[m] - r.tmin) * inv_scale : -1.0;
  }
  exp_table(s_table);
  __syncthreads();
  RowState at = state[i];  // (every thread reads back only what it wrote in s_time)
  for (int k = 0; k < grid.n; ++k) {
    const double T = grid.time(M, k);
    RowPoint out = {0.0, 0.0, 0.0, kNoRow};
    bool ok = !(F > 1.0 || T > hi * (1.0 + kTie));
    if (ok && T >= lo * (1.0 - kTie)) {
      if (flat) {
        out.kind = kEven;
        out.share = free_mass > 0.0 ? free_mass / (double)r.n_nb : 0.0;
      } else {
        const double target = fmin(fmax((T - A) / free_mass, r.tmin), r.tmax);
        const double sig = (target - r.tmin) / scale;
        double z = 1.0;
        RowState now = at;
        // moments of s under q ~ exp(-eta s)
        auto stats = [&](double e) {
          double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
          for (int m = threadIdx.x; m < M; m += blockDim.x) {
            const double s = s_time[m];
            if (s < 0.0) continue;
            const double w = table_exp(-e * s, s_table), ws = w * s, wss = ws * s;
            a0 += w;
            a1 += ws;
            a2 += wss;
            a3 += wss * s;
          }
          block_sum4(a0, a1, a2, a3, s_buf);
          z = a0;
          now.eta = e;
          now.mean = a1 / a0;
          now.var = a2 / a0 - now.mean * now.mean;
          now.third = a3 / a0 - now.mean * (3.0 * now.var + now.mean * now.mean);
        };
        double elo = -kEtaCap, ehi = kEtaCap;
        if (sig >= r.mean_lo) {
          stats(elo);
        } else if (sig <= r.mean_hi) {
          stats(ehi);
        } else {
          bool fresh = false;  // have the weights of this eta been added up?
          if (!(now.var > 0.0)) {
            stats(0.0);
            fresh = true;
          }
          for (int it = 0; it < 200; ++it) {  // steps kept inside a shrinking bracket
            const double gap = now.mean - sig;
            if (fresh && fabs(gap) <= 1e-15) break;
            if (gap > 0) elo = now.eta; else ehi = now.eta;
            const double slope = now.var * now.var - 0.5 * gap * now.third;
            double next = (now.var > 1e-300) ? now.eta + (slope > 0.5 * now.var * now.var ? gap * now.var / slope : gap / now.var) : 0.5 * (elo + ehi);
            if (!(next > elo && next < ehi)) next = 0.5 * (elo + ehi);
            if (fresh && (next == now.eta || ehi - elo <= 1e-15 * (1.0 + fabs(now.eta)))) break;
            // a step this short leaves an error of its square or less: below the rounding of the sums
            const bool last = fabs(next - now.eta) <= 1e-9 * (1.0 + fabs(now.eta)) && fabs(gap) <= 1e-9;
            stats(next);
            fresh = true;
            if (last) break;
          }
          at = now;
        }
        const double mean = now.mean, eta = now.eta;
        ok = fabs(mean - sig) <= 1e-9;
        out.kind = kTilted;
        out.eta = eta;
        out.share = free_mass / z;
      }
    } else if (ok) {
      const double pii = (lo - T) / (r.tmin - r.C);
      ok = !(pii > free_mass * (1.0 + kTie));
      out.kind = kFastest;
      out.pii = fmin(pii, free_mass);
      out.share = (free_mass - out.pii) / r.n_fast;
    }
    if (threadIdx.x == 0) {
      if (!ok) {
        out.kind = kNoRow;
        infeasible[k] = 1;
      }
      points[(size_t)k * M + i] = out;
    }
  }
  if (threadIdx.x == 0) state[i] = at;
}

// p_im of a link (i, m): f1 = d_im + d_mi.
__device__ __forceinline__ double row_entry(const RowInfo& r, const RowPoint& p, double ar, double f1, double t, double inv_scale, const double* s_table) {
  double p_im = ar * f1;
  if (p.kind == kTilted) p_im += p.share * table_exp(-p.eta * ((t - r.tmin) * inv_scale), s_table);
  else if (p.kind == kEven || t <= r.tmin * (1.0 + kTie)) p_im += p.share;
  return p_im;
}

// P at one grid point.
__global__ void __launch_bounds__(kRowThreads) store_rows_kernel(int M, const double* t, const uint8_t* adj, const RowInfo* info, double ar,
                                                                 const RowPoint* points, double* P) {
  __shared__ double s_table[kExpTable];
  exp_table(s_table);
  __syncthreads();
  const int i = blockIdx.x;
  const RowInfo r = info[i];
  const RowPoint p = points[i];
  const double inv_scale = 1.0 / (r.tmax - r.tmin);
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    const size_t at = (size_t)i * M + m;
    double v = m == i ? p.pii : 0.0;
    if (m != i && adj[at]) v = row_entry(r, p, ar, r.both ? 2.0 : (double)adj[at] + (double)adj[(size_t)m * M + i], t[at], inv_scale, s_table);
    P[at] = v;
  }
}

// How far the Rayleigh quotient v^T Y_P v of a unit vector (sum v_m = 0) lies below 1 at the points of a grid:
//   sum_{i < m} y_im (v_i - v_m)^2,  y_im (Eq. 22 with p_i = 1/M) = alpha rho/M [h(p_im) + h(p_mi)],
//   h(p) = (d_im+d_mi)/2 - alpha rho (d_im+d_mi)^2/(4p)  for p > 0,
// so every row adds up its own p_im and neither P nor Y need be stored (a pass over a stored P took 98 us per grid point of 4,096
// workers; this 27, bound by the fp64 pipe).  parts[k][i]: row i's share.
__global__ void __launch_bounds__(kRowThreads) row_quotient_kernel(int M, const double* t, const uint8_t* adj, const RowInfo* info,
                                                                   const PointGrid grid, const RowPoint* points, const double* v, double* parts) {
  extern __shared__ double s_time[];
  __shared__ double s_buf[33], s_table[kExpTable];
  exp_table(s_table);
  const int i = blockIdx.x;
  const RowInfo r = info[i];
  const double inv_scale = 1.0 / (r.tmax - r.tmin), vi = v[i], ar = grid.ar;
  for (int m = threadIdx.x; m < M; m += blockDim.x)
    s_time[m] = (m != i && adj[(size_t)i * M + m]) ? t[(size_t)i * M + m] : -1.0;  // (every thread reads back only what it wrote)
  __syncthreads();
  for (int k = 0; k < grid.n; ++k) {
    const RowPoint p = points[(size_t)k * M + i];
    double acc = 0.0;
    if (p.kind == kTilted && r.both) {  // the common form, its constants taken out: h(p) = 1 - ar / p, p = 2 ar + share exp(...)
      const double scaled = -p.eta * inv_scale, floor_im = 2.0 * ar;
      for (int m = threadIdx.x; m < M; m += blockDim.x) {
        const double tm = s_time[m];
        if (tm < 0.0) continue;
        const double d = vi - v[m];
        acc += fma(-ar, fast_reciprocal(fma(p.share, table_exp(scaled * (tm - r.tmin), s_table), floor_im)), 1.0) * (d * d);
      }
    } else if (p.kind != kNoRow) {
      for (int m = threadIdx.x; m < M; m += blockDim.x) {
        const double tm = s_time[m];
        if (tm < 0.0) continue;
        const double f1 = r.both ? 2.0 : 1.0 + (double)adj[(size_t)m * M + i];
        const double p_im = row_entry(r, p, ar, f1, tm, inv_scale, s_table), d = vi - v[m];
        if (p_im > 0.0) acc += (0.5 * f1 - ar * 0.25 * f1 * f1 * fast_reciprocal(p_im)) * d * d;
      }
    }
    acc = block_sum(acc, s_buf);
    if (threadIdx.x == 0) parts[(size_t)k * M + i] = ar / M * acc;
  }
}
// quotient[k] = 1 - sum of parts[k][.], in a fixed order.
__global__ void __launch_bounds__(256) quotient_sums_kernel(int M, const double* parts, double* quotient) {
  __shared__ double s_buf[33];
  double a = 0.0;
  for (int i = threadIdx.x; i < M; i += blockDim.x) a += parts[(size_t)blockIdx.x * M + i];
  a = block_sum(a, s_buf);
  if (threadIdx.x == 0) quotient[blockIdx.x] = 1.0 - a;
}

// Off-diagonal entries of Y_P (Eq. 22) with p_i = 1/M in the place of P: p_im gamma_im = (d_im+d_mi)/2,
// p_im gamma_im^2 = (d_im+d_mi)^2/(4 p_im).  y_im = y_mi needs p_im and p_mi: a CTA takes the tile (bi, bj) of the upper
// triangle and its mirror image, which nobody else looks at.  The diagonal is zero (the products with Y below never use it).
constexpr int kTile = 32;
struct TileIndex {
  int bi, bj;
};
// Tile number idx of the upper triangle of nb x nb tiles, row by row: row bi starts at bi nb - bi (bi - 1) / 2.
__device__ __forceinline__ TileIndex triangle_tile(long long idx, int nb) {
  auto start = [&](int b) { return (long long)b * nb - (long long)b * (b - 1) / 2; };
  const double e = 2.0 * nb + 1.0;
  int bi = (int)((e - sqrt(fmax(0.0, e * e - 8.0 * (double)idx))) * 0.5);
  bi = max(0, min(nb - 1, bi));
  while (bi > 0 && start(bi) > idx) --bi;
  while (bi + 1 < nb && start(bi + 1) <= idx) ++bi;
  return {bi, bi + (int)(idx - start(bi))};
}
__global__ void __launch_bounds__(256) y_tiles_kernel(int M, double* P, const uint8_t* adj, double ar) {
  __shared__ double s_mirror[kTile][kTile + 1];
  __shared__ uint8_t s_adj[kTile][kTile + 4];
  const int nb = (M + kTile - 1) / kTile;
  const TileIndex at = triangle_tile((long long)blockIdx.x, nb);
  const int bi = at.bi, bj = at.bj;
  const int c = threadIdx.x & (kTile - 1), r0 = threadIdx.x / kTile;
  const int i0 = bi * kTile, j0 = bj * kTile;
  for (int r = r0; r < kTile; r += 256 / kTile) {
    const int row = j0 + r, col = i0 + c;
    const bool in = row < M && col < M;
    s_mirror[r][c] = in ? P[(size_t)row * M + col] : 0.0;
    s_adj[r][c] = in ? adj[(size_t)row * M + col] : 0;
  }
  __syncthreads();
  double y[kTile * kTile / 256];
#pragma unroll
  for (int k = 0; k < kTile * kTile / 256; ++k) {
    const int r = r0 + k * (256 / kTile), i = i0 + r, m = j0 + c;
    y[k] = 0.0;
    if (i < M && m < M && i != m) {
      const double pim = P[(size_t)i * M + m], pmi = s_mirror[c][r];
      const double ds = (double)adj[(size_t)i * M + m] + (double)s_adj[c][r];
      double lin = 0.0, quad = 0.0;
      if (pim > 0.0) { lin += 0.5 * ds; quad += ds * ds / (4.0 * pim); }
      if (pmi > 0.0) { lin += 0.5 * ds; quad += ds * ds / (4.0 * pmi); }
      y[k] = (ar * lin - ar * ar * quad) / M;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kTile * kTile / 256; ++k) {
    const int r = r0 + k * (256 / kTile), i = i0 + r, m = j0 + c;
    if (i < M && m < M) P[(size_t)i * M + m] = y[k];
    s_mirror[c][r] = y[k];
  }
  __syncthreads();
  if (bi != bj)
    for (int r = r0; r < kTile; r += 256 / kTile) {
      const int row = j0 + r, col = i0 + c;
      if (row < M && col < M) P[(size_t)row * M + col] = s_mirror[r][c];
    }
}

// ---- Lanczos on the complement of the all-ones vector (fp64) -----------------------------------------
// Step k of the three-term recurrence in one launch, on B = Y - I.  Every CTA first finishes step k - 1 for
// itself: it adds the CTAs' shares of alpha = w . v_{k-1}, forms u = w - alpha v_{k-1} less its mean and
// v_k = u / |u| in its shared memory (M doubles; redundant, but a few
// microseconds against two more launches), and then multiplies its rows: w_i = (B v_k)_i - beta v_{k-1,i}.
// Rows of Y sum to 1, so (B v)_i = sum_m y_im (v_m - v_i): the diagonal is not needed, and what is summed
// has the size of the spectrum's spread (Y itself is close to I for many workers, and the rounding of
// numbers near 1 would swamp a beta of 1e-4 within a few steps).  No reorthogonalisation: the top of the
// spectrum converges all the same, copies of a converged value do not move it, and the component along
// the all-ones vector is taken out of every u.  Bound by reading Y (134 MB at M = 4096: 41 us per step with a CTA for every 16 rows, 256 of them,
// and 16-byte loads, 57 with one CTA per SM and 8-byte loads).
struct LanczosParams {
  int M, k;
  const double* Y;  // row-major; its block starts on 256 bytes
  double* V;        // [steps + 1][M]; row 0 is the start vector
  const double* w_in;
  double* w_out;
  const double* part_in;   // [gridDim.x]: shares of w . v of the previous step
  double* part_out;
  double* alpha;
  double* beta;
};
constexpr int kLanczosThreads = 512;
__global__ void __launch_bounds__(kLanczosThreads) lanczos_step_kernel(const LanczosParams p) {
  extern __shared__ __align__(16) double s_v[];
  __shared__ double s_buf[99];
  const int M = p.M, tid = threadIdx.x, T = blockDim.x;
  double beta_prev = 0.0;
  const double* v_prev = nullptr;
  if (p.k == 0) {
    for (int j = tid; j < M; j += T) s_v[j] = p.V[j];
    __syncthreads();
  } else {
    v_prev = p.V + (size_t)(p.k - 1) * M;
    double a = 0.0;
    for (int b = tid; b < (int)gridDim.x; b += T) a += __ldcg(p.part_in + b);
    a = block_sum(a, s_buf);
    double n2 = 0.0, s = 0.0, unused = 0.0;
    for (int j = tid; j < M; j += T) {
      const double u = p.w_in[j] - a * v_prev[j];
      s_v[j] = u;
      s += u;
      n2 += u * u;
    }
    block_sum3(n2, s, unused, s_buf);
    const double mean = s / M;  // (of u itself: what v_prev holds of it would come back scaled by alpha / beta)
    beta_prev = sqrt(fmax(0.0, n2 - s * mean));
    const double inv = beta_prev > 0.0 ? 1.0 / beta_prev : 0.0;
    for (int j = tid; j < M; j += T) {
      const double x = (s_v[j] - mean) * inv;
      s_v[j] = x;
      if (blockIdx.x == 0) p.V[(size_t)p.k * M + j] = x;
    }
    if (blockIdx.x == 0 && tid == 0) {
      p.alpha[p.k - 1] = a;
      p.beta[p.k - 1] = beta_prev;
    }
    __syncthreads();
  }
  const int lane = tid & 31, warp = tid >> 5, nw = T >> 5;
  double a = 0.0;
  for (int row = blockIdx.x * nw + warp; row < M; row += gridDim.x * nw) {
    const double* y = p.Y + (size_t)row * M;
    const double vi = s_v[row];
    double acc = 0.0;
    int j = lane;
    if ((M & 1) == 0) {  // pairs of columns (rows start on 16 bytes), eight loads in flight
      const double2* y2 = reinterpret_cast<const double2*>(y);
      const double2* v2 = reinterpret_cast<const double2*>(s_v);
      double other = 0.0;
      for (; 2 * (j + 224) < M; j += 256) {
        double2 in[8];
#pragma unroll
        for (int a = 0; a < 8; ++a)  // (volatile: issued one behind the other; left to itself the compiler keeps two in flight)
          asm volatile("ld.global.nc.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(in[a].x), "=d"(in[a].y) : "l"(y2 + j + 32 * a));
#pragma unroll
        for (int a = 0; a < 8; ++a) {
          const double2 v = v2[j + 32 * a];
          acc += in[a].x * (v.x - vi);
          other += in[a].y * (v.y - vi);
        }
      }
      for (; 2 * j < M; j += 32) {
        const double2 in = __ldg(y2 + j), v = v2[j];
        acc += in.x * (v.x - vi);
        other += in.y * (v.y - vi);
      }
      acc += other;
    } else {
#pragma unroll 8
      for (; j < M; j += 32) acc += y[j] * (s_v[j] - vi);
    }
    acc = warp_sum(acc);
    if (lane == 0) {
      const double w = acc - (p.k > 0 ? beta_prev * v_prev[row] : 0.0);
      p.w_out[row] = w;
      a += w * vi;
    }
  }
  a = block_sum(a, s_buf);
  if (tid == 0) p.part_out[blockIdx.x] = a;
}

// The coefficients of the last step (what the next step's launch would have written).
__global__ void __launch_bounds__(256) lanczos_tail_kernel(int k, int n_parts, const double* part, double* alpha) {
  __shared__ double s_buf[33];
  double a = 0.0;
  for (int b = threadIdx.x; b < n_parts; b += blockDim.x) a += part[b];
  a = block_sum(a, s_buf);
  if (threadIdx.x == 0) alpha[k] = a;
}

// probe = sum_k z_k V[k], centred and normalised: the Ritz vector, one CTA.
__global__ void __launch_bounds__(1024) ritz_vector_kernel(int M, int n, const double* V, const double* z, double* probe) {
  __shared__ double s_buf[33];
  double sum = 0.0;
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    double acc = 0.0;
    for (int k = 0; k < n; ++k) acc += z[k] * V[(size_t)k * M + j];
    probe[j] = acc;
    sum += acc;
  }
  const double mean = block_sum(sum, s_buf) / M;
  double n2 = 0.0;
  for (int j = threadIdx.x; j < M; j += blockDim.x) {
    const double x = probe[j] - mean;
    n2 += x * x;
  }
  const double inv = rsqrt(block_sum(n2, s_buf));
  for (int j = threadIdx.x; j < M; j += blockDim.x) probe[j] = (probe[j] - mean) * inv;
}

// ---- a policy change from link speeds -----------------------------------------------------------------
struct LinkStatus {
  unsigned long long n_min;  // bits of the least N_im (positive doubles compare as integers)
  int not_finite;
};

// Speeds -> link graph (a link needs a positive speed both ways) and N_im = 32 d / (s_im 1e9), in place.  A
// CTA takes a tile of the upper triangle and its mirror image.
__global__ void __launch_bounds__(256) links_kernel(int M, double d, double* st, uint8_t* adj, LinkStatus* status) {
  __shared__ double s_up[kTile][kTile + 1], s_low[kTile][kTile + 1];
  __shared__ double s_buf[33];
  const int nb = (M + kTile - 1) / kTile;
  const TileIndex at = triangle_tile((long long)blockIdx.x, nb);
  const int c = threadIdx.x & (kTile - 1), r0 = threadIdx.x / kTile;
  const int i0 = at.bi * kTile, j0 = at.bj * kTile;
  for (int r = r0; r < kTile; r += 256 / kTile) {
    s_up[r][c] = (i0 + r < M && j0 + c < M) ? st[(size_t)(i0 + r) * M + j0 + c] : 0.0;
    s_low[r][c] = (j0 + r < M && i0 + c < M) ? st[(size_t)(j0 + r) * M + i0 + c] : 0.0;
  }
  __syncthreads();
  double mn = INFINITY;
  bool bad = false;
  auto one = [&](int i, int m, double a, double b) {
    if (i >= M || m >= M) return;
    bad = bad || !isfinite(a);
    const bool link = i != m && a > 0.0 && b > 0.0;
    const double n = link ? 32.0 * d / (a * 1e9) : 0.0;
    adj[(size_t)i * M + m] = link;
    st[(size_t)i * M + m] = n;
    if (link) mn = fmin(mn, n);
  };
  for (int r = r0; r < kTile; r += 256 / kTile) {
    one(i0 + r, j0 + c, s_up[r][c], s_low[c][r]);
    if (at.bi != at.bj) one(j0 + r, i0 + c, s_low[r][c], s_up[c][r]);
  }
  mn = block_min(mn, s_buf);
  if (threadIdx.x == 0 && mn < INFINITY) atomicMin(&status->n_min, (unsigned long long)__double_as_longlong(mn));
  if (bad) status->not_finite = 1;
}

// t_ii = C = min N / 4, t_im = max{C, N_im} on links.
__global__ void __launch_bounds__(256) iteration_times_kernel(int M, double* t, const uint8_t* adj, const LinkStatus* status) {
  const double C = 0.25 * __longlong_as_double((long long)status->n_min);
  for (int i = blockIdx.x; i < M; i += gridDim.x)
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
      const size_t at = (size_t)i * M + m;
      if (i == m) t[at] = C;
      else if (adj[at]) t[at] = fmax(C, t[at]);
    }
}

// T_j = floor(cum_j 2^32 + 1/2) over the left-to-right prefix sums of a row of P (in this order: the draws
// are exact against these integers), non-decreasing, saturated, pinned to the top from the last positive
// entry on; and the pull weights.  A CTA takes eight rows, 128 columns at a time: a warp runs along its
// rows' sums, one row per lane, out of shared memory while the others convert the weights; all of them then turn sums into
// thresholds (with that in the chain 4,096 workers took 413 us).
constexpr int kTableRows = 8, kTableCols = 128, kTableThreads = 256;
__global__ void __launch_bounds__(kTableThreads) tables_kernel(int M, const double* P, const uint8_t* adj, double alpha_rho,
                                                               double pull_weight, uint32_t* thr, int32_t* last_nz, float* w) {
  __shared__ double s_p[kTableRows][kTableCols + 1];
  __shared__ double s_cum[kTableRows][kTableCols + 1];
  __shared__ int s_last[kTableRows];
  const int i0 = blockIdx.x * kTableRows, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int r = warp; r < kTableRows; r += kTableThreads / 32) {  // last positive entry, from the end
    const int i = i0 + r;
    int last = -1;
    if (i < M) {
      for (int base = (M - 1) & ~31; base >= 0; base -= 32) {
        const int j = base + lane;
        const unsigned hit = __ballot_sync(0xffffffffu, j < M && P[(size_t)i * M + j] > 0.0);
        if (hit) {
          last = base + 31 - __clz(hit);
          break;
        }
      }
      if (lane == 0) last_nz[i] = last;
    }
    if (lane == 0) s_last[r] = last;
  }
  double cum = 0.0;
  for (int j0 = 0; j0 < M; j0 += kTableCols) {
    __syncthreads();
    for (int k = tid; k < kTableRows * kTableCols; k += kTableThreads) {
      const int r = k / kTableCols, c = k % kTableCols, i = i0 + r, j = j0 + c;
      s_p[r][c] = (i < M && j < M) ? P[(size_t)i * M + j] : 0.0;
    }
    __syncthreads();
    if (warp == 0) {
      if (lane < kTableRows) {
#pragma unroll 16
        for (int c = 0; c < kTableCols; ++c) {
          cum += s_p[lane][c];
          s_cum[lane][c] = cum;
        }
      }
    } else {
      for (int k = tid - 32; k < kTableRows * kTableCols; k += kTableThreads - 32) {
        const int r = k / kTableCols, c = k % kTableCols, i = i0 + r, j = j0 + c;
        if (i >= M || j >= M) continue;
        const double p = s_p[r][c];
        float wv = 0.0f;
        if (i != j && p > 0.0) {
          const double dsum = 2.0 * (double)adj[(size_t)i * M + j];
          wv = pull_weight > 0.0 ? (float)pull_weight : (float)(alpha_rho * dsum / (2.0 * p));
        }
        w[(size_t)i * M + j] = wv;
      }
    }
    __syncthreads();
    for (int k = tid; k < kTableRows * kTableCols; k += kTableThreads) {
      const int r = k / kTableCols, c = k % kTableCols, i = i0 + r, j = j0 + c;
      if (i >= M || j >= M) continue;
      const double t = floor(s_cum[r][c] * 4294967296.0 + 0.5);  // (sums of entries >= 0 never decrease, nor do their roundings)
      thr[(size_t)i * M + j] = t > 4294967295.0 || j >= s_last[r] ? 0xFFFFFFFFu : (uint32_t)t;
    }
  }
}

}  // namespace

#include "netmax_policy_gpu_host.inc"
