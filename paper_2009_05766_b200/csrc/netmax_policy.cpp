// Host control plane of the NetMax simulator: the iteration-time model (Section II-B) and
// the communication-policy generator (Algorithm 3 with Eq. 8-14 and Eq. 22).
//
// Readings where the paper is silent or garbled:
//   * the grids are rho_k = k U_rho / K and t_bar_r = U - (R - r)(U - L)/R;
//   * U_rho = min(0.5/alpha, (1 - 1e-6) / (alpha max_i sum_{m != i}(d_im + d_mi))), because
//     beyond it the floors of Eq. 11 alone exceed a row sum of one;
//   * L = max_i (alpha rho / M) sum_{m != i} t_im (d_im + d_mi)   (Eq. 25-26);
//   * d_ii = 1 for selectability and t_ii = C_i; Eq. 11 is taken closed;
//   * the LP (Eq. 14) decouples by row and its optimum is not unique: when p_ii = 0 is
//     feasible the row is floor + (1 - sum floors) * q with q_m ~ exp(-eta t_im) matched to
//     the required mean time (the maximum-entropy optimum); otherwise p_ii is the least
//     value that meets the time constraint and the remainder goes to the fastest peer(s);
//   * with every row meeting Eq. 10, p_i = 1/M (Lemma 1), which Y_P uses directly;
//   * eps = 1e-3; infeasible grid points are skipped; ties keep the earlier grid point.
//
// The same search for pull rules with a constant weight w (the section on extending existing
// decentralised PSGD approaches), netmax_policy_generate_fixed_weight:
//   * E[D^T D] for D = I + w e_i (e_m - e_i)^T has y_im = (w - w^2)(p_i p_im + p_m p_mi), so the
//     replacement of Eq. 11 ("every y_im on a link is positive") reads p_im + p_mi > 0; it is taken
//     closed with a floor phi on both directions of every link, and phi takes rho's place in the
//     outer loop (phi_k = k U_phi / K, U_phi where the floors alone fill a row);
//   * Y_P is doubly stochastic only if, besides Eq. 10 (p_i = 1/M), the columns of P sum to 1
//     (row sums of Y_P are 1 + w (sum_m p_m p_mi - p_i sum_m p_im)): an added constraint that couples
//     the rows of the LP;
//   * the optimum is again not unique; the reading is p_ii = 0 and the maximum-entropy P above the
//     floors, p_im = phi + A_i B_m exp(-eta_i t_im), found by alternating scalings: rows (A_i and
//     eta_i from the row's sum and mean time), then columns (B_m from the column sums); the inner
//     grid takes the midpoints of R cells of [L, U].
#include "../../include/netmax.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <mutex>
#include <thread>
#include <vector>

#include "netmax_policy.h"

namespace {

constexpr double kEtaCap = 600.0;
constexpr double kTie = 1e-12;
constexpr double kEps = 1e-3;

int fail(int code, const std::string& msg) {
  netmax::set_global_error(msg);
  return code;
}

template <typename Body>
void parallel_for(int n, int min_parallel, const Body& body) {
  netmax::parallel_rows(n, min_parallel, [&](int64_t a, int64_t b) { body((int)a, (int)b); });
}

// ---- vector helpers: eight doubles at a time, compiled for the instruction sets a host may have -----
typedef double vec8 __attribute__((vector_size(64)));
typedef int64_t ivec8 __attribute__((vector_size(64)));
#if defined(__x86_64__) && defined(__GNUC__)
#define NM_CLONES __attribute__((target_clones("avx512f", "avx2", "default")))
#else
#define NM_CLONES
#endif

// Sums over j < n (n a multiple of 8) of w, w s and w s^2 with w_j = g_j exp(-eta s_j); w is kept in q.
// The exponential is Cody and Waite's: x = k ln 2 + r with the multiple taken off in two parts, a Taylor
// polynomial of degree 13 on |r| <= ln 2 / 2 (remainder below 5e-18), and k added to the exponent
// (|eta s| <= 600 keeps the result a normal number).  The row solves spend their time here.
NM_CLONES void tilt_sums(const double* s, const double* g, int n, double eta, double* q, double* z, double* a, double* b) {
  vec8 vz = {}, va = {}, vb = {};
  const double kLog2e = 1.4426950408889634074, kLn2Hi = 6.93147180369123816490e-01, kLn2Lo = 1.90821492927058770002e-10;
  const double kShift = 6755399441055744.0;  // 1.5 2^52: adding it rounds to an integer in the low mantissa bits
  for (int j = 0; j < n; j += 8) {
    vec8 sv, gv;
    __builtin_memcpy(&sv, s + j, 64);
    __builtin_memcpy(&gv, g + j, 64);
    const vec8 x = sv * -eta;
    const vec8 t = x * kLog2e + kShift;
    const vec8 kf = t - kShift;
    const vec8 r = (x - kf * kLn2Hi) - kf * kLn2Lo;
    vec8 p = r * (1.0 / 6227020800.0) + (1.0 / 479001600.0);
    p = p * r + (1.0 / 39916800.0);
    p = p * r + (1.0 / 3628800.0);
    p = p * r + (1.0 / 362880.0);
    p = p * r + (1.0 / 40320.0);
    p = p * r + (1.0 / 5040.0);
    p = p * r + (1.0 / 720.0);
    p = p * r + (1.0 / 120.0);
    p = p * r + (1.0 / 24.0);
    p = p * r + (1.0 / 6.0);
    p = p * r + 0.5;
    p = p * r + 1.0;
    p = p * r + 1.0;
    ivec8 e, bits;
    __builtin_memcpy(&e, &t, 64);
    __builtin_memcpy(&bits, &p, 64);
    bits += e << 52;
    vec8 w;
    __builtin_memcpy(&w, &bits, 64);
    w *= gv;
    __builtin_memcpy(q + j, &w, 64);
    const vec8 ws = w * sv;
    vz += w;
    va += ws;
    vb += ws * sv;
  }
  double tz = 0, ta = 0, tb = 0;
  for (int l = 0; l < 8; ++l) { tz += vz[l]; ta += va[l]; tb += vb[l]; }
  *z = tz; *a = ta; *b = tb;
}

NM_CLONES double dot(const double* x, const double* y, int n) {
  vec8 acc = {};
  int j = 0;
  for (; j + 8 <= n; j += 8) {
    vec8 a, b;
    __builtin_memcpy(&a, x + j, 64);
    __builtin_memcpy(&b, y + j, 64);
    acc += a * b;
  }
  double t = 0.0;
  for (; j < n; ++j) t += x[j] * y[j];
  for (int l = 0; l < 8; ++l) t += acc[l];
  return t;
}

// y += c x
NM_CLONES void axpy(double* y, const double* x, double c, int n) {
  int j = 0;
  for (; j + 8 <= n; j += 8) {
    vec8 a, b;
    __builtin_memcpy(&a, y + j, 64);
    __builtin_memcpy(&b, x + j, 64);
    a += b * c;
    __builtin_memcpy(y + j, &a, 64);
  }
  for (; j < n; ++j) y[j] += c * x[j];
}

// One row of the LP, apart from the grid point.  s, g, q have n8 entries, n rounded up to a multiple of
// eight: entries beyond n weigh nothing.
struct Row {
  std::vector<int> nb;           // neighbours m != i
  std::vector<double> t, f1;     // their iteration times and d_im + d_mi
  std::vector<double> s, g;      // times mapped to [0, 1]; 1 for a neighbour, 0 for filling
  double C = 0, tmin = 0, tmax = 0, sum_f1 = 0, sum_f1t = 0;
  double mean_lo = 0, mean_hi = 0;  // mean s at the ends of the bracket, eta = -+kEtaCap
  bool flat = false;             // all links equally fast
};

void finish_row(Row& r) {
  const size_t n = r.nb.size(), n8 = (n + 7) / 8 * 8;
  const double scale = r.tmax - r.tmin;
  r.flat = !(scale > kTie * r.tmax);
  if (r.flat) return;
  r.s.assign(n8, 0.0);
  r.g.assign(n8, 0.0);
  for (size_t j = 0; j < n; ++j) {
    r.s[j] = (r.t[j] - r.tmin) / scale;
    r.g[j] = 1.0;
  }
  std::vector<double> q(n8);
  double z, a, b;
  tilt_sums(r.s.data(), r.g.data(), (int)n8, -kEtaCap, q.data(), &z, &a, &b);
  r.mean_lo = a / z;
  tilt_sums(r.s.data(), r.g.data(), (int)n8, kEtaCap, q.data(), &z, &a, &b);
  r.mean_hi = a / z;
}

// Exponential tilt: q_m ~ exp(-eta s_m), s in [0,1], with mean s equal to sig.  The mean is decreasing
// in eta; Newton steps are kept inside a shrinking bracket.  *eta is the start (the neighbouring grid
// point's solution: two or three steps from this one's) and receives the solution; q holds the
// unnormalised weights and *z their sum.
bool tilt(const Row& row, double sig, double* eta_io, double* q, double* z_out) {
  const int n8 = (int)row.s.size();
  double z = 1.0, mean = 0.0, var = 0.0;
  auto stats = [&](double eta) {
    double a, b;
    tilt_sums(row.s.data(), row.g.data(), n8, eta, q, &z, &a, &b);
    mean = a / z;
    var = b / z - mean * mean;
  };
  double lo = -kEtaCap, hi = kEtaCap, eta = *eta_io;
  if (sig >= row.mean_lo) {
    stats(eta = lo);
  } else if (sig <= row.mean_hi) {
    stats(eta = hi);
  } else {
    if (!(eta > lo && eta < hi)) eta = 0.0;
    stats(eta);
    for (int it = 0; it < 200; ++it) {
      const double gap = mean - sig;
      if (std::fabs(gap) <= 1e-15) break;
      if (gap > 0) lo = eta; else hi = eta;
      double next = (var > 1e-300) ? eta + gap / var : 0.5 * (lo + hi);
      if (!(next > lo && next < hi)) next = 0.5 * (lo + hi);
      if (next == eta || hi - lo <= 1e-15 * (1.0 + std::fabs(eta))) break;
      // a Newton step this short leaves an error of its square: below the rounding of the sums
      const bool last = std::fabs(next - eta) <= 1e-9 * (1.0 + std::fabs(eta)) && std::fabs(gap) <= 1e-9;
      eta = next;
      stats(eta);
      if (last) break;
    }
  }
  *eta_io = eta;
  *z_out = z;
  return std::fabs(mean - sig) <= 1e-9;
}

// One row of the LP at (rho, T = M t_bar).  Returns false when the row is infeasible.
bool solve_row(const Row& row, int i, int M, double ar /* alpha rho */, double T, double* eta, double* q, double* out) {
  const size_t n = row.nb.size();
  const double F = ar * row.sum_f1;
  if (F > 1.0) return false;
  const double free_mass = 1.0 - F;
  const double A = ar * row.sum_f1t;
  const double lo = A + free_mass * row.tmin, hi = A + free_mass * row.tmax;
  if (T > hi * (1.0 + kTie)) return false;
  if (n + 1 < (size_t)M) std::fill(out, out + M, 0.0);
  out[i] = 0.0;
  if (T >= lo * (1.0 - kTie)) {
    if (free_mass <= 0.0) {
      for (size_t j = 0; j < n; ++j) out[row.nb[j]] = ar * row.f1[j];
      return true;
    }
    if (row.flat) {
      for (size_t j = 0; j < n; ++j) out[row.nb[j]] = ar * row.f1[j] + free_mass * (1.0 / (double)n);
      return true;
    }
    const double target = std::min(std::max((T - A) / free_mass, row.tmin), row.tmax);
    double z = 1.0;
    if (!tilt(row, (target - row.tmin) / (row.tmax - row.tmin), eta, q, &z)) return false;
    const double f = free_mass / z;
    for (size_t j = 0; j < n; ++j) out[row.nb[j]] = ar * row.f1[j] + f * q[j];
    return true;
  }
  double pii = (lo - T) / (row.tmin - row.C);
  if (pii > free_mass * (1.0 + kTie)) return false;
  pii = std::min(pii, free_mass);
  int fastest = 0;
  for (size_t j = 0; j < n; ++j) fastest += (row.t[j] <= row.tmin * (1.0 + kTie));
  for (size_t j = 0; j < n; ++j) {
    const bool fast = row.t[j] <= row.tmin * (1.0 + kTie);
    out[row.nb[j]] = ar * row.f1[j] + (fast ? (free_mass - pii) / fastest : 0.0);
  }
  out[i] = pii;
  return true;
}

// ---- eigenvalues of symmetric tridiagonal matrices ------------------------------------------------
// How many eigenvalues of the tridiagonal matrix (diagonal d[0..m), squares of the off-diagonal e2) lie
// below x: the negative pivots of T - x I (Sturm's sequence).
int count_below(const double* d, const double* e2, int m, double x) {
  int count = 0;
  double q = d[0] - x;
  for (int i = 0;;) {
    if (std::fabs(q) < 1e-300) q = -1e-300;
    count += q < 0.0;
    if (++i == m) break;
    q = d[i] - x - e2[i - 1] / q;
  }
  return count;
}

// The eigenvalue number `index` (ascending, from 0), by bisection to neighbouring doubles.
double tridiagonal_eigenvalue(const double* d, const double* e, int m, int index) {
  std::vector<double> e2(m);
  double lo = INFINITY, hi = -INFINITY;
  for (int i = 0; i < m; ++i) {
    const double off = (i > 0 ? std::fabs(e[i - 1]) : 0.0) + (i + 1 < m ? std::fabs(e[i]) : 0.0);
    lo = std::min(lo, d[i] - off);
    hi = std::max(hi, d[i] + off);
    if (i + 1 < m) e2[i] = e[i] * e[i];
  }
  const double pad = 1e-15 * std::max(std::fabs(lo), std::fabs(hi)) + 1e-300;
  lo -= pad;
  hi += pad;
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (!(mid > lo && mid < hi)) break;
    if (count_below(d, e2.data(), m, mid) > index) hi = mid; else lo = mid;
  }
  return 0.5 * (lo + hi);
}

// An eigenvector of the tridiagonal matrix for the eigenvalue lambda: inverse iteration, two steps, with
// row exchanges in the elimination.
void tridiagonal_eigenvector(const double* d, const double* e, int m, double lambda, std::vector<double>& z) {
  z.assign(m, 0.0);
  if (m == 1) { z[0] = 1.0; return; }
  std::vector<double> u0(m), u1(m, 0.0), u2(m, 0.0), l(m, 0.0);
  std::vector<uint8_t> swapped(m, 0);
  double tiny = 0.0;  // a pivot that stands for zero: the matrix's rounding
  for (int i = 0; i < m; ++i) tiny = std::max(tiny, std::fabs(d[i]) + (i + 1 < m ? std::fabs(e[i]) : 0.0));
  tiny = 1e-16 * tiny + 1e-300;
  double a = d[0] - lambda, b = e[0];  // the current row: diagonal, superdiagonal
  for (int i = 0; i + 1 < m; ++i) {
    const double c = e[i], dn = d[i + 1] - lambda, bn = i + 2 < m ? e[i + 1] : 0.0;
    if (std::fabs(c) > std::fabs(a)) {
      swapped[i] = 1;
      l[i] = a / c;
      u0[i] = c; u1[i] = dn; u2[i] = bn;
      a = b - l[i] * dn;
      b = -l[i] * bn;
    } else {
      if (std::fabs(a) < tiny) a = tiny;
      l[i] = c / a;
      u0[i] = a; u1[i] = b;
      a = dn - l[i] * b;
      b = bn;
    }
  }
  u0[m - 1] = std::fabs(a) < tiny ? tiny : a;
  for (int j = 0; j < m; ++j) z[j] = 1.0 + 0.37 * (j % 5);
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = 0; i + 1 < m; ++i) {
      if (swapped[i]) std::swap(z[i], z[i + 1]);
      z[i + 1] -= l[i] * z[i];
    }
    for (int i = m - 1; i >= 0; --i) {
      double v = z[i];
      if (i + 1 < m) v -= u1[i] * z[i + 1];
      if (i + 2 < m) v -= u2[i] * z[i + 2];
      z[i] = v / u0[i];
    }
    double big = 0.0;
    for (double v : z) big = std::max(big, std::fabs(v));
    for (double& v : z) v /= big;
  }
}

// Takes the component along the all-ones vector out of v and normalises it.
void centre(std::vector<double>& v) {
  const int M = (int)v.size();
  double mean = 0.0, nrm = 0.0;
  for (double x : v) mean += x;
  mean /= M;
  for (double& x : v) { x -= mean; nrm += x * x; }
  nrm = std::sqrt(nrm);
  if (!(nrm > 0.0)) { v.clear(); return; }
  for (double& x : v) x /= nrm;
}

// Second largest eigenvalue of the symmetric doubly stochastic Y: the largest eigenvalue of Y
// restricted to the complement of the all-ones vector.  Householder's reduction to tridiagonal form and
// bisection for small M; Lanczos with full reorthogonalisation otherwise.  vec (may be NULL) receives an
// approximate eigenvector in that complement.
double second_eigenvalue(const std::vector<double>& Y, int M, std::vector<double>* vec, bool parallel) {
  if (M <= 96) {
    std::vector<double> A(Y), d(M), e(M, 0.0), w(M), scale(M, 0.0);
    // column k is reduced with the reflection I - scale[k] v v^T; v stays in row k of A, from k + 1 on
    for (int k = 0; k + 2 < M; ++k) {
      double* v = A.data() + (size_t)k * M;  // row k = column k of the symmetric matrix
      const int n = M - k - 1;
      const double norm = std::sqrt(dot(v + k + 1, v + k + 1, n));
      d[k] = v[k];
      if (!(norm > 0.0)) continue;
      const double alpha = v[k + 1] > 0.0 ? -norm : norm;
      e[k] = alpha;
      const double beta = 1.0 / (norm * norm - alpha * v[k + 1]);  // 2 / v^T v once alpha is taken off
      v[k + 1] -= alpha;
      scale[k] = beta;
      for (int i = k + 1; i < M; ++i) w[i] = beta * dot(A.data() + (size_t)i * M + k + 1, v + k + 1, n);
      const double half = 0.5 * beta * dot(w.data() + k + 1, v + k + 1, n);
      axpy(w.data() + k + 1, v + k + 1, -half, n);
      for (int i = k + 1; i < M; ++i) {
        double* row = A.data() + (size_t)i * M;
        axpy(row + k + 1, w.data() + k + 1, -v[i], n);
        axpy(row + k + 1, v + k + 1, -w[i], n);
      }
    }
    if (M >= 2) {
      d[M - 2] = A[(size_t)(M - 2) * M + M - 2];
      e[M - 2] = A[(size_t)(M - 2) * M + M - 1];
    }
    d[M - 1] = A[(size_t)(M - 1) * M + M - 1];
    const double lam = tridiagonal_eigenvalue(d.data(), e.data(), M, M - 2);
    if (vec) {
      std::vector<double>& z = *vec;
      tridiagonal_eigenvector(d.data(), e.data(), M, lam, z);
      for (int k = M - 3; k >= 0; --k) {
        const double* v = A.data() + (size_t)k * M + k + 1;
        axpy(z.data() + k + 1, v, -scale[k] * dot(v, z.data() + k + 1, M - k - 1), M - k - 1);
      }
      centre(z);
    }
    return lam;
  }
  auto matvec = [&](const std::vector<double>& v, std::vector<double>& out) {
    double mean = 0.0;
    for (int j = 0; j < M; ++j) mean += v[j];
    mean /= M;
    parallel_for(M, parallel ? 512 : M + 1, [&](int a, int b) {
      for (int i = a; i < b; ++i) out[i] = dot(Y.data() + (size_t)i * M, v.data(), M) - mean;  // (Y - 11^T/M) v
    });
  };
  const int max_steps = std::min(M - 1, 300);
  std::vector<std::vector<double>> V;
  std::vector<double> alpha, beta, v(M), wv(M);
  uint64_t lcg = 0x9E3779B97F4A7C15ull;
  for (int j = 0; j < M; ++j) {
    lcg = lcg * 6364136223846793005ull + 1442695040888963407ull;
    v[j] = (double)(lcg >> 11) / 9007199254740992.0 - 0.5;
  }
  centre(v);
  double best = 0.0;
  for (int step = 0; step < max_steps; ++step) {
    V.push_back(v);
    matvec(v, wv);
    alpha.push_back(dot(wv.data(), v.data(), M));
    for (int pass = 0; pass < 2; ++pass)  // full reorthogonalisation, twice
      for (const auto& u : V) axpy(wv.data(), u.data(), -dot(wv.data(), u.data(), M), M);
    const double b = std::sqrt(dot(wv.data(), wv.data(), M));
    const int m = (int)alpha.size();
    if ((m % 10 == 0) || b < 1e-13 || step == max_steps - 1) {
      const double top = tridiagonal_eigenvalue(alpha.data(), beta.data(), m, m - 1);
      const bool settled = std::fabs(top - best) <= 1e-13 * std::max(1.0, std::fabs(top));
      best = top;
      if (b < 1e-13 || (settled && m >= 20)) break;
    }
    beta.push_back(b);
    for (int j = 0; j < M; ++j) v[j] = wv[j] / b;
  }
  if (vec) {
    std::vector<double> z;
    tridiagonal_eigenvector(alpha.data(), beta.data(), (int)alpha.size(), best, z);
    vec->assign(M, 0.0);
    for (size_t k = 0; k < z.size(); ++k) axpy(vec->data(), V[k].data(), z[k], M);
    centre(*vec);
  }
  return best;
}

}  // namespace

namespace netmax {
double tridiagonal_top_eigenvalue(const std::vector<double>& alpha, const std::vector<double>& beta) {
  return tridiagonal_eigenvalue(alpha.data(), beta.data(), (int)alpha.size(), (int)alpha.size() - 1);
}
void tridiagonal_top_vector(const std::vector<double>& alpha, const std::vector<double>& beta, double lambda, std::vector<double>& z) {
  tridiagonal_eigenvector(alpha.data(), beta.data(), (int)alpha.size(), lambda, z);
}
}  // namespace netmax

extern "C" {

int netmax_iteration_times(int32_t M, int64_t d, const double* speed, double* t_out, uint8_t* adj_out) try {
  if (M < 2 || d < 1 || !speed || !t_out || !adj_out) return fail(NETMAX_INVALID_ARG, "iteration_times: bad argument");
  // (by blocks of columns, so that the transposed entries are read a cache line at a time; rows over threads)
  constexpr int kBlock = 64;
  std::vector<double> row_min(M, INFINITY);
  std::atomic<bool> finite{true};
  netmax::parallel_rows(M, 512, [&](int64_t r0, int64_t r1) {
    for (int64_t ib = r0; ib < r1; ib += kBlock)
      for (int64_t mb = 0; mb < M; mb += kBlock)
        for (int64_t i = ib; i < std::min(r1, ib + kBlock); ++i)
          for (int64_t m = mb; m < std::min<int64_t>(M, mb + kBlock); ++m) {
            const size_t at = (size_t)i * M + m;
            const double a = speed[at], b = speed[(size_t)m * M + i];
            if (!std::isfinite(a)) finite = false;
            const bool link = (i != m) && a > 0.0 && b > 0.0;
            adj_out[at] = link ? 1 : 0;
            t_out[at] = link ? 32.0 * (double)d / (a * 1e9) : 0.0;   // N_im: a full fp32 replica over the link
            if (link) row_min[i] = std::min(row_min[i], t_out[at]);
          }
  });
  if (!finite) return fail(NETMAX_INVALID_ARG, "iteration_times: link speed is not finite");
  const double nmin = *std::min_element(row_min.begin(), row_min.end());
  if (!std::isfinite(nmin)) return fail(NETMAX_NOT_CONNECTED, "iteration_times: no link has a positive speed");
  const double C = 0.25 * nmin;   // C_i: computation is the short part of an iteration
  netmax::parallel_rows(M, 512, [&](int64_t r0, int64_t r1) {
    for (int64_t i = r0; i < r1; ++i)
      for (int64_t m = 0; m < M; ++m) {
        const size_t at = (size_t)i * M + m;
        if (i == m) t_out[at] = C;
        else if (adj_out[at]) t_out[at] = std::max(C, t_out[at]);   // t_im = max{C_i, N_im}
      }
  });
  return NETMAX_OK;
} NM_CATCH(fail)

int netmax_policy_generate(int32_t M, const double* t, const uint8_t* adj, double lr, int32_t K, int32_t R,
                           double* prob_out, double* rho_out, double* info_out) {
  return netmax_policy_generate_ex(M, t, adj, lr, K, R, 0.0, prob_out, rho_out, info_out);
}

int netmax_policy_generate_ex(int32_t M, const double* t, const uint8_t* adj, double lr, int32_t K, int32_t R,
                              double rho_upper, double* prob_out, double* rho_out, double* info_out) try {
  if (M < 2 || !t || !adj || !prob_out || !rho_out || !(lr > 0.0) || K < 1 || R < 1)
    return fail(NETMAX_INVALID_ARG, "policy_generate: bad argument");
  std::vector<Row> rows(M);
  double max_f1 = 0.0, U_time = INFINITY;
  for (int i = 0; i < M; ++i) {
    Row& r = rows[i];
    r.C = t[(size_t)i * M + i];
    r.tmin = INFINITY;
    r.tmax = 0.0;
    for (int m = 0; m < M; ++m) {
      if (m == i || !adj[(size_t)i * M + m]) continue;
      const double tm = t[(size_t)i * M + m];
      if (!(tm > 0.0) || !std::isfinite(tm)) return fail(NETMAX_INVALID_ARG, "policy_generate: iteration time on a link is not positive");
      const double f1 = (double)adj[(size_t)i * M + m] + (double)adj[(size_t)m * M + i];
      r.nb.push_back(m);
      r.t.push_back(tm);
      r.f1.push_back(f1);
      r.sum_f1 += f1;
      r.sum_f1t += f1 * tm;
      r.tmin = std::min(r.tmin, tm);
      r.tmax = std::max(r.tmax, tm);
    }
    if (r.nb.empty()) return fail(NETMAX_NOT_CONNECTED, "policy_generate: a worker has no neighbour");
    if (!(r.C < r.tmin)) return fail(NETMAX_INVALID_ARG, "policy_generate: t_ii must be below every t_im");
    max_f1 = std::max(max_f1, r.sum_f1);
    U_time = std::min(U_time, r.tmax / M);
  }
  const double U_rho = rho_upper > 0.0 ? rho_upper : std::min(0.5 / lr, (1.0 - 1e-6) / (lr * max_f1));

  for (Row& r : rows) finish_row(r);

  // The grid.  lambda_2 is what costs: it is only computed where it can matter.  With v orthogonal to the
  // all-ones vector the Rayleigh quotient v^T Y v = 1 - sum_{i<m} y_im (v_i - v_m)^2 bounds lambda_2 from
  // below, and t_conv grows with lambda_2; with v the eigenvector of the best point so far nearly every
  // other point is ruled out by that bound (with a margin far above its rounding).  The values of rho are
  // shared out over threads, each of which walks its t_bar grid in order, every row starting from the
  // solution of the previous grid point; the outcome does not depend on how the threads are timed.
  struct Best {
    std::vector<double> P;
    double tconv = INFINITY, rho = 0, lam = 0, tbar = 0;
    int k = 0, r = 0;
  };
  const double work_ns = (double)K * R * M * M * 12.0;
  const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
  const bool by_rows = M >= 1024;  // a copy of P and Y per thread would be too much: threads share a grid point instead
  int n_threads = by_rows ? 1 : (int)std::min<double>(std::min<double>(std::min<unsigned>(hw, netmax::kMaxThreads), K), 1.0 + work_ns / 4e5);
  std::mutex mu;
  std::vector<double> probe;             // eigenvector of the best point so far (guarded by mu)
  double probe_tconv = INFINITY;
  int next_k = 1;
  auto walk = [&](std::vector<Best>& found) {
    std::vector<double> P((size_t)M * M), Y, eta(M), v, vec;
    std::vector<std::vector<double>> q(by_rows ? M : 1);  // scratch of solve_row
    for (auto& buf : q) buf.resize((size_t)M + 8);
    double v_tconv = INFINITY;
    std::vector<uint8_t> ok(M);
    std::vector<double> share(M);
    for (;;) {
      int k;
      {
        std::lock_guard<std::mutex> lock(mu);
        k = next_k++;
      }
      if (k > K) return;
      const double rho = k * U_rho / K, ar = lr * rho;
      double L = 0.0;
      for (int i = 0; i < M; ++i) L = std::max(L, ar / M * rows[i].sum_f1t);
      if (!(U_time > L)) continue;
      const double delta = (U_time - L) / R;
      std::fill(eta.begin(), eta.end(), 0.0);
      Best best;
      for (int r = 1; r <= R; ++r) {
        const double tbar = U_time - (R - r) * delta, T = M * tbar;
        bool feasible = true;
        if (by_rows) {
          parallel_for(M, 256, [&](int a, int b) {
            for (int i = a; i < b; ++i)
              ok[i] = solve_row(rows[i], i, M, ar, T, &eta[i], q[i].data(), P.data() + (size_t)i * M) ? 1 : 0;
          });
          feasible = std::find(ok.begin(), ok.end(), (uint8_t)0) == ok.end();
        } else {
          for (int i = 0; i < M && feasible; ++i)
            feasible = solve_row(rows[i], i, M, ar, T, &eta[i], q[0].data(), P.data() + (size_t)i * M);
        }
        if (!feasible) continue;
        {
          std::lock_guard<std::mutex> lock(mu);
          if (probe_tconv < v_tconv) { v = probe; v_tconv = probe_tconv; }
        }
        // Y_P (Eq. 22) with p_i = 1/M: p_im gamma_im = (d_im+d_mi)/2, p_im gamma_im^2 = (d_im+d_mi)^2/(4 p_im)
        auto y_of = [&](int i, int m) {
          const double pim = P[(size_t)i * M + m], pmi = P[(size_t)m * M + i];
          const double ds = (double)adj[(size_t)i * M + m] + (double)adj[(size_t)m * M + i];
          double lin = 0.0, quad = 0.0;
          if (pim > 0.0) { lin += 0.5 * ds; quad += ds * ds / (4.0 * pim); }
          if (pmi > 0.0) { lin += 0.5 * ds; quad += ds * ds / (4.0 * pmi); }
          return (ar * lin - ar * ar * quad) / M;
        };
        if (!v.empty()) {
          parallel_for(M, by_rows ? 256 : M + 1, [&](int a, int b) {
            for (int i = a; i < b; ++i) {
              double acc = 0.0;
              for (int m = i + 1; m < M; ++m) acc += y_of(i, m) * ((v[i] - v[m]) * (v[i] - v[m]));
              share[i] = acc;
            }
          });
          double rq = 1.0;
          for (int i = 0; i < M; ++i) rq -= share[i];
          if (rq > 0.0 && rq < 1.0 && tbar * std::log(kEps) / std::log(rq) > v_tconv * (1.0 + 1e-9)) continue;
        }
        Y.resize((size_t)M * M);
        parallel_for(M, by_rows ? 256 : M + 1, [&](int a, int b) {
          for (int i = a; i < b; ++i) {
            double rowsum = 0.0;
            for (int m = 0; m < M; ++m) {
              if (m == i) continue;
              const double y = y_of(i, m);
              Y[(size_t)i * M + m] = y;
              rowsum += y;
            }
            Y[(size_t)i * M + i] = 1.0 - rowsum;
          }
        });
        const double lam2 = second_eigenvalue(Y, M, &vec, by_rows);
        if (!(lam2 > 0.0 && lam2 < 1.0)) continue;
        const double tconv = tbar * std::log(kEps) / std::log(lam2);
        if (!vec.empty() && tconv < v_tconv) {
          v = vec;
          v_tconv = tconv;
          std::lock_guard<std::mutex> lock(mu);
          if (tconv < probe_tconv) { probe = vec; probe_tconv = tconv; }
        }
        if (best.P.empty() || tconv < best.tconv * (1.0 - 1e-12)) {
          best.P = P;
          best.tconv = tconv;
          best.rho = rho;
          best.lam = lam2;
          best.tbar = tbar;
          best.k = k;
          best.r = r;
        }
      }
      if (!best.P.empty()) {
        // (of the thread's own rhos only candidates are kept: none that an earlier one of them beats)
        if (found.empty() || best.tconv < found.back().tconv * (1.0 - 1e-12)) found.push_back(std::move(best));
        if (found.size() > 2) found.erase(found.begin(), found.end() - 2);
      }
    }
  };
  std::vector<std::vector<Best>> found(n_threads);
  netmax::on_threads(n_threads, [&](int th) { walk(found[th]); });
  std::vector<const Best*> order;
  for (const auto& list : found)
    for (const Best& b : list) order.push_back(&b);
  std::sort(order.begin(), order.end(), [](const Best* a, const Best* b) { return a->k < b->k; });
  const Best* best = nullptr;
  for (const Best* b : order)  // grid order: ties keep the earlier point
    if (!best || b->tconv < best->tconv * (1.0 - 1e-12)) best = b;
  if (!best) return fail(NETMAX_INFEASIBLE, "policy_generate: no feasible (rho, t_bar) grid point");
  std::copy(best->P.begin(), best->P.end(), prob_out);
  *rho_out = best->rho;
  if (info_out) {
    info_out[0] = best->lam;
    info_out[1] = best->tbar;
    info_out[2] = best->tconv;
    info_out[3] = best->k;
    info_out[4] = best->r;
  }
  return NETMAX_OK;
} NM_CATCH(fail)

}  // extern "C"


// ---- constant pull weight -----------------------------------------------------------------------
namespace {

// The maximum-entropy P above the floor phi with zero diagonal, rows and columns summing to 1 and
// sum_m t_im p_im = T in every row.  Residual r = p - phi on links: r_im = A_i B_m exp(-eta_i s_im)
// with s the iteration times mapped to [0, 1].  Rows first (eta_i by a bracketed Newton iteration
// on the row's mean time, then A_i from its sum), then columns (B_m); repeated until every
// constraint holds to 1e-12.  Returns false when the constraints cannot be met.
bool solve_fixed_weight(int M, const double* t, const uint8_t* adj, double phi, double T, std::vector<double>& P) {
  std::vector<std::vector<int>> nb(M);
  std::vector<double> rows(M), cols(M, 1.0), tau(M);
  double tmin = INFINITY, tmax = 0.0;
  for (int i = 0; i < M; ++i)
    for (int m = 0; m < M; ++m)
      if (m != i && adj[(size_t)i * M + m]) {
        nb[i].push_back(m);
        tmin = std::min(tmin, t[(size_t)i * M + m]);
        tmax = std::max(tmax, t[(size_t)i * M + m]);
        cols[m] -= phi;
      }
  const bool homogeneous = tmax - tmin <= kTie * tmax;  // all links equally fast: the time constraint only says T = t
  if (homogeneous && std::fabs(T - tmin) > 1e-9 * tmax) return false;
  const double scale = homogeneous ? INFINITY : tmax - tmin;  // (t - tmin) / scale = 0 on every link then
  bool floors_fill = true;
  for (int i = 0; i < M; ++i) {
    rows[i] = 1.0 - phi * (double)nb[i].size();
    if (rows[i] < -1e-15) return false;
    double floor_time = 0.0;
    for (int m : nb[i]) floor_time += t[(size_t)i * M + m];
    tau[i] = homogeneous ? 0.0 : (T - phi * floor_time - tmin * rows[i]) / scale;  // target of sum_m s_im r_im
    if (rows[i] > 1e-15) floors_fill = false;
  }
  P.assign((size_t)M * M, 0.0);
  auto finish = [&](const std::vector<double>& r) {
    double worst = 0.0;
    std::vector<double> colsum(M, 0.0);
    for (int i = 0; i < M; ++i) {
      double sum = 0.0, time = 0.0;
      for (int m : nb[i]) {
        const double p = phi + r[(size_t)i * M + m];
        P[(size_t)i * M + m] = p;
        sum += p;
        time += p * t[(size_t)i * M + m];
        colsum[m] += p;
      }
      worst = std::max(worst, std::max(std::fabs(sum - 1.0), std::fabs(time - T) / tmax));
    }
    for (int m = 0; m < M; ++m) worst = std::max(worst, std::fabs(colsum[m] - 1.0));
    return worst <= 1e-9;
  };
  std::vector<double> r((size_t)M * M, 0.0);
  if (floors_fill) return finish(r);
  for (int i = 0; i < M; ++i)
    if (tau[i] < -1e-12 || tau[i] > rows[i] * (1.0 + 1e-12)) return false;

  std::vector<double> A(M, 1.0), B(M, 1.0), eta(M, 0.0), wgt(M);
  double err_mark = INFINITY;
  for (int sweep = 0; sweep < 20000; ++sweep) {
    // rows: weights B_m exp(-eta s_im); their mean s must equal tau_i / rows_i
    double row_change = 0.0;
    for (int i = 0; i < M; ++i) {
      if (!(rows[i] > 1e-15)) { A[i] = 0.0; continue; }
      const double sig = std::min(std::max(tau[i] / rows[i], 0.0), 1.0);
      auto stats = [&](double e, double& z, double& mean, double& var) {
        double a = 0.0, b = 0.0;
        z = 0.0;
        for (int m : nb[i]) {
          const double sv = (t[(size_t)i * M + m] - tmin) / scale;
          const double w = B[m] * std::exp(-e * sv);
          z += w;
          a += w * sv;
          b += w * sv * sv;
        }
        mean = a / z;
        var = b / z - mean * mean;
      };
      double lo = -kEtaCap, hi = kEtaCap, e = eta[i], z, mean, var;
      stats(lo, z, mean, var);
      if (sig >= mean) {
        e = lo;
      } else {
        stats(hi, z, mean, var);
        if (sig <= mean) {
          e = hi;
        } else {
          stats(e, z, mean, var);
          for (int it = 0; it < 200; ++it) {
            const double gap = mean - sig;
            if (std::fabs(gap) <= 1e-15) break;
            if (gap > 0) lo = e; else hi = e;
            double next = (var > 1e-300) ? e + gap / var : 0.5 * (lo + hi);
            if (!(next > lo && next < hi)) next = 0.5 * (lo + hi);
            if (next == e || hi - lo <= 1e-15 * (1.0 + std::fabs(e))) break;
            e = next;
            stats(e, z, mean, var);
          }
        }
      }
      stats(e, z, mean, var);
      row_change = std::max(row_change, std::fabs(e - eta[i]));
      eta[i] = e;
      A[i] = rows[i] / z;
    }
    // columns: B_m from the column sums
    double col_err = 0.0;
    std::fill(wgt.begin(), wgt.end(), 0.0);
    for (int i = 0; i < M; ++i)
      for (int m : nb[i]) wgt[m] += A[i] * std::exp(-eta[i] * (t[(size_t)i * M + m] - tmin) / scale);
    for (int m = 0; m < M; ++m) {
      if (!(wgt[m] > 0.0)) continue;
      const double next = std::max(cols[m], 0.0) / wgt[m];
      col_err = std::max(col_err, std::fabs(next - B[m]) * wgt[m]);   // column sum before the rescaling, off by this much
      B[m] = next;
    }
    if (col_err <= 1e-13 && row_change <= 1e-12) break;
    // a target outside the reachable set never settles: give up when 500 sweeps did not halve the misfit
    // (a grid point that converges more slowly than that counts as infeasible)
    if (sweep % 500 == 0) {
      if (sweep > 0 && col_err > 0.5 * err_mark) break;
      err_mark = col_err;
    }
  }
  for (int i = 0; i < M; ++i)
    for (int m : nb[i]) r[(size_t)i * M + m] = A[i] * B[m] * std::exp(-eta[i] * (t[(size_t)i * M + m] - tmin) / scale);
  return finish(r);
}

}  // namespace

extern "C" {

int netmax_policy_fixed_weight_at(int32_t M, const double* t, const uint8_t* adj, double floor, double t_bar, double* prob_out) try {
  if (M < 2 || !t || !adj || !prob_out || !(floor >= 0.0) || !(t_bar > 0.0) || !std::isfinite(floor) || !std::isfinite(t_bar))
    return fail(NETMAX_INVALID_ARG, "policy_fixed_weight_at: bad argument");
  std::vector<double> P;
  if (!solve_fixed_weight(M, t, adj, floor, M * t_bar, P))
    return fail(NETMAX_INFEASIBLE, "policy_fixed_weight_at: no P meets the floors, the row and column sums and the mean iteration time");
  std::copy(P.begin(), P.end(), prob_out);
  return NETMAX_OK;
} NM_CATCH(fail)

int netmax_policy_generate_fixed_weight(int32_t M, const double* t, const uint8_t* adj, double pull_weight, int32_t K,
                                        int32_t R, double floor_upper, double* prob_out, double* floor_out, double* info_out) try {
  if (M < 2 || !t || !adj || !prob_out || !floor_out || !(pull_weight > 0.0 && pull_weight < 1.0) || K < 1 || R < 1)
    return fail(NETMAX_INVALID_ARG, "policy_generate_fixed_weight: bad argument");
  int max_deg = 0;
  for (int i = 0; i < M; ++i) {
    int deg = 0;
    for (int m = 0; m < M; ++m) {
      if (m == i || !adj[(size_t)i * M + m]) continue;
      if (!adj[(size_t)m * M + i]) return fail(NETMAX_INVALID_ARG, "policy_generate_fixed_weight: the link graph must be symmetric");
      const double tm = t[(size_t)i * M + m];
      if (!(tm > 0.0) || !std::isfinite(tm)) return fail(NETMAX_INVALID_ARG, "policy_generate_fixed_weight: iteration time on a link is not positive");
      ++deg;
    }
    if (deg == 0) return fail(NETMAX_NOT_CONNECTED, "policy_generate_fixed_weight: a worker has no neighbour");
    max_deg = std::max(max_deg, deg);
  }
  const double U_phi = floor_upper > 0.0 ? floor_upper : (1.0 - 1e-6) / max_deg;
  const double w = pull_weight;
  std::vector<double> P, Y((size_t)M * M), bestP;
  double best_tconv = INFINITY, best_phi = 0, best_lam = 0, best_tbar = 0;
  int best_k = 0, best_r = 0;
  for (int k = 1; k <= K; ++k) {
    const double phi = k * U_phi / K;
    // range of the rows' mean time: floors plus all of the remainder on the fastest / slowest link
    double L = 0.0, U = INFINITY;
    bool rows_ok = true;
    for (int i = 0; i < M; ++i) {
      double sum_t = 0.0, tmin = INFINITY, tmax = 0.0;
      int deg = 0;
      for (int m = 0; m < M; ++m) {
        if (m == i || !adj[(size_t)i * M + m]) continue;
        const double tm = t[(size_t)i * M + m];
        sum_t += tm;
        tmin = std::min(tmin, tm);
        tmax = std::max(tmax, tm);
        ++deg;
      }
      const double rest = 1.0 - phi * deg;
      if (rest < -1e-15) rows_ok = false;
      L = std::max(L, (phi * sum_t + rest * tmin) / M);
      U = std::min(U, (phi * sum_t + rest * tmax) / M);
    }
    if (!rows_ok || !(U >= L)) continue;
    for (int r = 1; r <= R; ++r) {
      const double tbar = L + (r - 0.5) * (U - L) / R;  // cell midpoints: the end points are degenerate vertices
      if (!solve_fixed_weight(M, t, adj, phi, M * tbar, P)) continue;
      // E[D^T D] with p_i = 1/M (Eq. 10 holds by construction)
      for (int i = 0; i < M; ++i) {
        double pulls = 0.0, pulled = 0.0;
        for (int m = 0; m < M; ++m) {
          if (m == i) continue;
          const double pim = P[(size_t)i * M + m], pmi = P[(size_t)m * M + i];
          Y[(size_t)i * M + m] = (w - w * w) * (pim + pmi) / M;
          pulls += pim;
          pulled += pmi;
        }
        Y[(size_t)i * M + i] = 1.0 - (2.0 * w - w * w) * pulls / M + w * w * pulled / M;
      }
      const double lam2 = second_eigenvalue(Y, M, nullptr, true);
      if (!(lam2 > 0.0 && lam2 < 1.0)) continue;
      const double tconv = tbar * std::log(kEps) / std::log(lam2);
      if (bestP.empty() || tconv < best_tconv * (1.0 - 1e-12)) {
        bestP = P;
        best_tconv = tconv;
        best_phi = phi;
        best_lam = lam2;
        best_tbar = tbar;
        best_k = k;
        best_r = r;
      }
    }
  }
  if (bestP.empty()) return fail(NETMAX_INFEASIBLE, "policy_generate_fixed_weight: no feasible (floor, t_bar) grid point");
  std::copy(bestP.begin(), bestP.end(), prob_out);
  *floor_out = best_phi;
  if (info_out) {
    info_out[0] = best_lam;
    info_out[1] = best_tbar;
    info_out[2] = best_tconv;
    info_out[3] = best_k;
    info_out[4] = best_r;
  }
  return NETMAX_OK;
} NM_CATCH(fail)

}  // extern "C"
