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

#include "netmax_policy.h"

namespace {

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

// Sums of three values over the CTA, returned to every thread.  s_buf: 99 doubles.
__device__ void block_sum3(double& a, double& b, double& c, double* s_buf) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  a = warp_sum(a);
  b = warp_sum(b);
  c = warp_sum(c);
  __syncthreads();
  if (lane == 0) {
    s_buf[warp] = a;
    s_buf[33 + warp] = b;
    s_buf[66 + warp] = c;
  }
  __syncthreads();
  if (warp < 3) {
    double t = lane < nw ? s_buf[33 * warp + lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) s_buf[33 * warp + 32] = t;
  }
  __syncthreads();
  a = s_buf[32];
  b = s_buf[65];
  c = s_buf[98];
}

// What the host looks at after every grid point.
struct PointResult {
  double rq;        // Rayleigh quotient of the probe vector
  int infeasible;   // some row of the LP has no solution
};

// One row of the LP at (alpha rho, T = M t_bar); an infeasible row raises out->infeasible.
// Bound by fp64 exponentials: the row's times, mapped to [0, 1], stay in shared memory (-1: no link) for
// all Newton steps, which start from the previous grid point's solution (eta[i]) and so are two or three.
__global__ void __launch_bounds__(kRowThreads) row_solve_kernel(int M, const double* t, const uint8_t* adj, const RowInfo* info,
                                                                double ar, double T, double* P, double* eta_io, PointResult* out) {
  extern __shared__ double s_time[];
  __shared__ double s_buf[99];
  const int i = blockIdx.x;
  const RowInfo r = info[i];
  const double* ti = t + (size_t)i * M;
  const uint8_t* ai = adj + (size_t)i * M;
  double* pi = P + (size_t)i * M;
  const double F = ar * r.sum_f1;
  const double free_mass = 1.0 - F, A = ar * r.sum_f1t;
  const double lo = A + free_mass * r.tmin, hi = A + free_mass * r.tmax;
  if (F > 1.0 || T > hi * (1.0 + kTie)) {
    if (threadIdx.x == 0) out->infeasible = 1;
    return;
  }
  auto f1_of = [&](int m) { return r.both ? 2.0 : (double)ai[m] + (double)adj[(size_t)m * M + i]; };
  if (T >= lo * (1.0 - kTie)) {
    const double scale = r.tmax - r.tmin;
    const bool flat = !(scale > kTie * r.tmax) || free_mass <= 0.0;
    double eta = 0.0, z = (double)r.n_nb;
    if (!flat) {
      const double target = fmin(fmax((T - A) / free_mass, r.tmin), r.tmax);
      const double sig = (target - r.tmin) / scale, inv_scale = 1.0 / scale;
      for (int m = threadIdx.x; m < M; m += blockDim.x) s_time[m] = (m != i && ai[m]) ? (ti[m] - r.tmin) * inv_scale : -1.0;
      // mean and variance of s under q ~ exp(-eta s)  (every thread reads back only what it wrote)
      double mean, var;
      auto stats = [&](double e) {
        double a0 = 0, a1 = 0, a2 = 0;
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
          const double s = s_time[m];
          if (s < 0.0) continue;
          const double w = exp(-e * s);
          a0 += w;
          a1 += w * s;
          a2 += w * s * s;
        }
        block_sum3(a0, a1, a2, s_buf);
        z = a0;
        mean = a1 / a0;
        var = a2 / a0 - mean * mean;
      };
      double elo = -kEtaCap, ehi = kEtaCap;
      if (sig >= r.mean_lo) {
        stats(eta = elo);
      } else if (sig <= r.mean_hi) {
        stats(eta = ehi);
      } else {
        eta = eta_io[i];
        stats(eta);
        for (int it = 0; it < 200; ++it) {  // Newton steps kept inside a shrinking bracket
          const double gap = mean - sig;
          if (fabs(gap) <= 1e-15) break;
          if (gap > 0) elo = eta; else ehi = eta;
          double next = (var > 1e-300) ? eta + gap / var : 0.5 * (elo + ehi);
          if (!(next > elo && next < ehi)) next = 0.5 * (elo + ehi);
          if (next == eta || ehi - elo <= 1e-15 * (1.0 + fabs(eta))) break;
          // a Newton step this short leaves an error of its square: below the rounding of the sums
          const bool last = fabs(next - eta) <= 1e-9 * (1.0 + fabs(eta)) && fabs(gap) <= 1e-9;
          eta = next;
          stats(eta);
          if (last) break;
        }
        __syncthreads();  // (every thread has read eta_io[i])
        if (threadIdx.x == 0) eta_io[i] = eta;
      }
      if (threadIdx.x == 0 && !(fabs(mean - sig) <= 1e-9)) out->infeasible = 1;
    }
    const double share = flat ? (free_mass > 0.0 ? free_mass / (double)r.n_nb : 0.0) : free_mass / z;
    for (int m = threadIdx.x; m < M; m += blockDim.x) {
      double p = 0.0;
      if (m != i && ai[m]) p = ar * f1_of(m) + (flat ? share : share * exp(-eta * s_time[m]));
      pi[m] = p;
    }
    return;
  }
  double pii = (lo - T) / (r.tmin - r.C);
  if (pii > free_mass * (1.0 + kTie)) {
    if (threadIdx.x == 0) out->infeasible = 1;
    return;
  }
  pii = fmin(pii, free_mass);
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    double p = 0.0;
    if (m == i) p = pii;
    else if (ai[m]) p = ar * f1_of(m) + (ti[m] <= r.tmin * (1.0 + kTie) ? (free_mass - pii) / r.n_fast : 0.0);
    pi[m] = p;
  }
}

// Off-diagonal entries of Y_P (Eq. 22) with p_i = 1/M: p_im gamma_im = (d_im+d_mi)/2,
// p_im gamma_im^2 = (d_im+d_mi)^2/(4 p_im).  y_im = y_mi needs p_im and p_mi: a CTA takes the tile (bi, bj)
// of the upper triangle and its mirror image, so that P is read once and coalesced.
//   kStore  writes both tiles of Y, with a zero diagonal (the products with Y below never use it);
//   else    sums y_im (v_i - v_m)^2 over the tile: 1 minus the sum over all tiles is the Rayleigh quotient
//           v^T Y v of a unit vector.  The last CTA adds the tiles in order and leaves the result in out->rq.
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
template <bool kStore>
__global__ void __launch_bounds__(256) y_tiles_kernel(int M, const double* P, const uint8_t* adj, double ar, double* Y, const double* v,
                                                      double* partial, unsigned int* ticket, PointResult* out) {
  __shared__ double s_mirror[kTile][kTile + 1];
  __shared__ uint8_t s_adj[kTile][kTile + 4];
  __shared__ double s_buf[33];
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
  double acc = 0.0;
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
      if (!kStore && i < m) {
        const double d = v[i] - v[m];
        acc += y[k] * d * d;
      }
    }
  }
  if (kStore) {
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kTile * kTile / 256; ++k) {
      const int r = r0 + k * (256 / kTile), i = i0 + r, m = j0 + c;
      if (i < M && m < M) Y[(size_t)i * M + m] = y[k];
      s_mirror[c][r] = y[k];
    }
    __syncthreads();
    if (bi != bj)
      for (int r = r0; r < kTile; r += 256 / kTile) {
        const int row = j0 + r, col = i0 + c;
        if (row < M && col < M) Y[(size_t)row * M + col] = s_mirror[r][c];
      }
    return;
  }
  acc = block_sum(acc, s_buf);
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = acc;
    __threadfence();
    s_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double sum = 0.0;
  for (unsigned int k = threadIdx.x; k < gridDim.x; k += blockDim.x) sum += __ldcg(partial + k);
  sum = block_sum(sum, s_buf);
  if (threadIdx.x == 0) {
    out->rq = 1.0 - sum;
    *ticket = 0u;
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
// the all-ones vector is taken out of every u.  Bound by reading Y (134 MB at M = 4096).
struct LanczosParams {
  int M, k;
  const double* Y;
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
  extern __shared__ double s_v[];
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
    for (; j + 96 < M; j += 128) {  // four loads in flight
      const double y0 = y[j], y1 = y[j + 32], y2 = y[j + 64], y3 = y[j + 96];
      acc += y0 * (s_v[j] - vi);
      acc += y1 * (s_v[j + 32] - vi);
      acc += y2 * (s_v[j + 64] - vi);
      acc += y3 * (s_v[j + 96] - vi);
    }
    for (; j < M; j += 32) acc += y[j] * (s_v[j] - vi);
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
// entry on; and the pull weights.  A CTA takes 32 rows, 64 columns at a time: one warp runs along its 32
// rows' sums, one row per lane, out of shared memory while the others convert the weights.
constexpr int kTableRows = 32, kTableCols = 64, kTableThreads = 256;
__global__ void __launch_bounds__(kTableThreads) tables_kernel(int M, const double* P, const uint8_t* adj, double alpha_rho,
                                                               double pull_weight, uint32_t* thr, int32_t* last_nz, float* w) {
  __shared__ double s_p[kTableRows][kTableCols + 1];
  __shared__ uint32_t s_t[kTableRows][kTableCols + 1];
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
  unsigned long long prev = 0;
  for (int j0 = 0; j0 < M; j0 += kTableCols) {
    __syncthreads();
    for (int k = tid; k < kTableRows * kTableCols; k += kTableThreads) {
      const int r = k / kTableCols, c = k % kTableCols, i = i0 + r, j = j0 + c;
      s_p[r][c] = (i < M && j < M) ? P[(size_t)i * M + j] : 0.0;
    }
    __syncthreads();
    if (warp == 0) {
      const int last = s_last[lane];
      for (int c = 0; c < kTableCols; ++c) {
        cum += s_p[lane][c];
        unsigned long long t = (unsigned long long)floor(cum * 4294967296.0 + 0.5);
        t = t > prev ? t : prev;
        if (t > 0xFFFFFFFFull || j0 + c >= last) t = 0xFFFFFFFFull;
        s_t[lane][c] = (uint32_t)t;
        prev = t;
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
      if (i < M && j < M) thr[(size_t)i * M + j] = s_t[r][c];
    }
  }
}

}  // namespace

#include "netmax_policy_gpu_host.inc"
