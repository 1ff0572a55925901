"""The policy search's own exponential and reciprocal, as the device computes them, against 80-bit ones on the host: over the whole range that
they are for, at the ends of it, at zero and on both sides of every boundary between entries of the exponential's table.  Bounds: the table's
entry and the last multiply-add round once each and r's rounding and the polynomial's add less than half a unit (2 units in the last
place); Newton's second step leaves the rounding of its own sum (1)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_05766_b200", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include "netmax_fp64.cuh"
using namespace netmax;

__global__ void both(const double* x, const double* y, double* ex, double* ry, int n) {
  __shared__ double table[kExpTable];
  exp_table(table);
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  ex[i] = table_exp(x[i], table);
  ry[i] = fast_reciprocal(y[i]);
}
static double units(double got, long double want) {  // of the last place of the wanted value
  int e;
  std::frexp((double)want, &e);
  return (double)(fabsl((long double)got - want) / ldexpl(1.0L, e - 53));
}
int main() {
  std::vector<double> x{0.0, -0.0, 1e-300, -1e-18, 600.0, -600.0}, y;
  for (int k = -13848; k <= 13848; ++k) {
    const double edge = (k + 0.5) * 0.69314718055994531 / 16.0;
    for (double v : {std::nextafter(edge, -1e9), edge, std::nextafter(edge, 1e9)})
      if (std::fabs(v) <= 600.0) x.push_back(v);
  }
  std::mt19937_64 gen(7);
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  while (x.size() < (1u << 19)) x.push_back((x.size() & 1 ? 600.0 : 1.0) * u(gen));
  for (int e = -60; e <= 60; ++e) for (double m : {1.0, std::nextafter(1.0, 2.0), std::nextafter(2.0, 1.0)}) y.push_back(std::ldexp(m, e));
  while (y.size() < x.size()) y.push_back(std::exp(20.0 * u(gen)));
  const int n = (int)x.size();
  double *dx, *dy, *de, *dr;
  for (double** p : {&dx, &dy, &de, &dr}) if (cudaMalloc(p, n * 8) != cudaSuccess) return 2;
  cudaMemcpy(dx, x.data(), n * 8, cudaMemcpyHostToDevice);
  cudaMemcpy(dy, y.data(), n * 8, cudaMemcpyHostToDevice);
  both<<<(n + 255) / 256, 256>>>(dx, dy, de, dr, n);
  std::vector<double> ex(n), ry(n);
  cudaMemcpy(ex.data(), de, n * 8, cudaMemcpyDeviceToHost);
  if (cudaMemcpy(ry.data(), dr, n * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  double worst_e = 0.0, worst_r = 0.0;
  for (int i = 0; i < n; ++i) {
    worst_e = std::fmax(worst_e, units(ex[i], expl((long double)x[i])));
    worst_r = std::fmax(worst_r, units(ry[i], 1.0L / (long double)y[i]));
  }
  std::printf("%.4f %.4f\n", worst_e, worst_r);
  return 0;
}
"""


def test_exponential_and_reciprocal_against_long_double(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2009_05766_b200 import build
    src, exe = tmp_path / "fp64.cu", tmp_path / "fp64"
    src.write_text(PROGRAM)
    subprocess.run([build._nvcc(), "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert done.returncode == 0, done.stdout + done.stderr
    exponential, reciprocal = (float(v) for v in done.stdout.split())
    assert exponential <= 2.0 and reciprocal <= 1.0, done.stdout
