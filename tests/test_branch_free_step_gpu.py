"""The register-resident kernel's step without branches, at the node counts where a
lane or a whole warp is left without a node, and the branch-free square root."""
import os
import subprocess

import numpy as np
import pytest

from oracle import game_pdhg as GO
from oracle import lax_pdhg as O
from paper_1803_01215_gb300 import build_lib, workloads as W

torch = pytest.importorskip("torch")

from gpu_common import gpu, value_err  # noqa: E402

pytestmark = pytest.mark.gpu

SQRT = r"""
#include <cstdio>
#include "hj_internal.cuh"
__global__ void k(unsigned long long* bad) {
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < (1ull << 32); i += step) {
    const float x = __uint_as_float((unsigned)i), r = sqrtf(x), b = hj::sqrt_rn_nb(x);
    if (r != r ? b == b : __float_as_uint(r) != __float_as_uint(b)) atomicAdd(bad, 1ull);
  }
}
int main() {
  unsigned long long *d, h = 1;
  cudaMalloc(&d, 8);
  cudaMemset(d, 0, 8);
  k<<<1520, 256>>>(d);
  cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost);
  printf("%llu %d\n", h, (int)cudaDeviceSynchronize());
}
"""


def test_branch_free_root_is_sqrtf_on_every_argument(tmp_path):
    src, exe = tmp_path / "root.cu", tmp_path / "root"
    src.write_text(SQRT)
    subprocess.run([build_lib.nvcc_path(), *build_lib.ARCH, *build_lib.NVCC_FLAGS, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True, env=dict(os.environ))
    assert out.stdout.split() == ["0", "0"]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("N", [1, 2, 31, 32, 33, 64, 65, 96, 97, 128])
def test_quadcopter_fixed_iterations_at_the_group_edges(N, precision):
    """K = 40 iterations element by element: FP64 to 1e-10; FP32 to 40 steps' rounding
    (2^-24 times a few operations each, iterates up to 4) with a factor 10: 1e-4."""
    w = W.quadcopter(B=7, seed=5, N=N, t=0.5)
    K = 40
    g = gpu(w, precision, tol=0.0, max_iter=K, check_every=K)
    o = O.solve(w, tol=0.0, max_iter=K, check_every=K)
    tol = 1e-10 if precision == "fp64" else 1e-4
    assert np.all(g["iters"] == K)
    assert np.max(np.abs(g["traj_x"] - o["x"])) <= tol
    assert np.max(np.abs(g["traj_p"] - o["p"])) <= tol
    assert np.max(value_err(g["V"], o["V"])) <= (1e-9 if precision == "fp64" else 1e-4)
    np.testing.assert_array_equal(g["traj_x"][:, N], w["xq"].astype(g["traj_x"].dtype))   # x_N = x


@pytest.mark.parametrize("d1", [1, 3])
def test_game_split_fixed_at_compile_time_and_not(d1):
    """d1 = 1 runs the instantiation with the split folded in, d1 = 3 the general one."""
    w = W.game_norms(d=7, B=9, seed=12)
    w["N"], w["t"] = 6, np.full(9, 6 * W.EIK_DELTA)
    w["dyn"] = np.array(w["dyn"])
    w["dyn"][0] = d1
    g = gpu(w, "fp64", tol=0.0, max_iter=150, check_every=150)
    o = GO.solve_game(w, tol=0.0, max_iter=150, check_every=150)
    assert np.max(np.abs(g["traj_x"] - o["x"])) <= 1e-10
    assert np.max(np.abs(g["traj_p"] - o["p"])) <= 1e-10
    assert np.max(value_err(g["V"], o["V"])) <= 1e-9
