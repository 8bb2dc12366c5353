"""The Taylor-table tanh against the host's extended-precision tanhl (113 bits where long
double is binary128, else 64): at most 1 ulp, the bound that CUDA documents for its own
tanh.  Its terms: half an ulp of the last addition, half an ulp of c_1 b, and c_1's own
rounding, which are together below 1 wherever c_1 b is smaller than the result's binade
(from row 2 on) and were found at 0.87 in the one row where it is not."""
import os
import subprocess

import pytest

from paper_1803_01215_gb300 import build_lib

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include "hj_internal.cuh"
#include "tanh64.cuh"
__global__ void k(const double* x, double* y, int n) {
  extern __shared__ double tab[];
  hj::tanh_taylor_table(tab, threadIdx.x, blockDim.x);
  __syncthreads();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) y[i] = hj::tanh_taylor(x[i], tab);
}
int main() {
  // over [0, 20], magnitudes from 2^-60 up, and densely where the table's error is largest
  const int n = 3 << 19;
  std::vector<double> x(n), y(n);
  std::mt19937_64 g(11);
  for (int i = 0; i < n; ++i) {
    const double u = (double)(g() >> 11) * 0x1p-53;
    x[i] = i % 3 == 0 ? 20.0 * u : i % 3 == 1 ? std::exp2(70.0 * u - 60.0) : std::exp2(4.0 * u - 5.0);
    if (i & 1) x[i] = -x[i];
  }
  x[0] = 0.531649; x[1] = 0.2175; x[2] = 0.0312715; x[3] = 19.0625;
  double *dx, *dy;
  cudaMalloc(&dx, n * 8); cudaMalloc(&dy, n * 8);
  cudaMemcpy(dx, x.data(), n * 8, cudaMemcpyHostToDevice);
  k<<<152, 256, hj::kTanhRows * hj::kTanhRow * 8>>>(dx, dy, n);
  cudaMemcpy(y.data(), dy, n * 8, cudaMemcpyDeviceToHost);
  double w = 0.0, at = 0.0;
  for (int i = 0; i < n; ++i) {
    const long double t = tanhl((long double)x[i]);
    int e;
    std::frexp((double)t, &e);
    const double err = std::fabs((double)(((long double)y[i] - t) / std::ldexp(1.0, e - 53)));
    if (!(err <= w)) { w = err; at = x[i]; }
  }
  printf("%.4f %.17g %d\n", w, at, (int)cudaDeviceSynchronize());
}
"""


def test_table_tanh_is_within_one_ulp(tmp_path):
    src, exe = tmp_path / "tanh.cu", tmp_path / "tanh"
    src.write_text(SRC)
    subprocess.run([build_lib.nvcc_path(), *build_lib.ARCH, *build_lib.NVCC_FLAGS, str(src), "-o", str(exe)], check=True)
    worst, at, err = subprocess.run([str(exe)], capture_output=True, text=True, check=True,
                                    env=dict(os.environ)).stdout.split()
    print(f"tanh: largest error {worst} ulp at {at}")
    assert int(err) == 0
    assert float(worst) <= 1.0
