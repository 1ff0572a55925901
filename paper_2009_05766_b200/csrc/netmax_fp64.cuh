// Double precision functions of the policy search's row kernels, which the fp64 pipe bounds.
#pragma once
#include <cuda_runtime.h>

namespace netmax {

// exp(x) for |x| <= 600 by a table of powers of two (Tang, "Table-driven implementation of the exponential function"): x =
// (16 e + j) ln 2 / 16 + r with the multiple taken off in two parts, exp(r) by its Taylor polynomial of degree 7 (|r| <= ln 2 / 32:
// remainder below 2e-18), times 2^(j/16) out of shared memory, with e added to the exponent.  Sixteen doubles fill the 32 banks once,
// so no access conflicts.  Twelve operations of the fp64 pipe, which is what bounds the row kernels (see row_solve_kernel).
constexpr int kExpTable = 16;
__device__ __forceinline__ void exp_table(double* s_table) {  // (before a __syncthreads)
  if (threadIdx.x < kExpTable) s_table[threadIdx.x] = exp2((double)threadIdx.x / kExpTable);
}
__device__ __forceinline__ double table_exp(double x, const double* s_table) {
  const double shift = 6755399441055744.0;  // 1.5 2^52: adding it rounds to an integer in the low mantissa bits
  const double t = fma(x, 23.083120654223414, shift), k = t - shift;  // 16 / ln 2
  const int n = __double2loint(t);
  double r = fma(k, -0x1.62e42fefp-5, x);          // ln 2 / 16: its leading 32 bits (k has 14), and the rest
  r = fma(k, -0x1.473de6af278edp-38, r);
  double q = fma(r, 1.0 / 5040.0, 1.0 / 720.0);
  q = fma(q, r, 1.0 / 120.0);
  q = fma(q, r, 1.0 / 24.0);
  q = fma(q, r, 1.0 / 6.0);
  q = fma(q, r, 0.5);
  q = fma(q, r, 1.0) * r;
  const double p = s_table[n & (kExpTable - 1)];
  const double v = fma(p, q, p);
  return __hiloint2double(__double2hiint(v) + ((n >> 4) << 20), __double2loint(v));
}

// 1 / x for x well inside the range of normal numbers: Newton's iteration on the hardware's approximation (about 20 bits, then
// 40, then rounding).
__device__ __forceinline__ double fast_reciprocal(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

}  // namespace netmax
