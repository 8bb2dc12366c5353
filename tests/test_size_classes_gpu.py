"""Kernels that are chosen or laid out by size, at the edges of their classes.

Where two instantiations do the same arithmetic (a uniform batch without node guards
against a ragged plan with them; a tile's columns past N against a smaller launch), a
fixed number of iterations gives the same bits.  FP64 against the oracle: 1e-10 after
40 iterations.  The Taylor-table tanh: CUDA documents 1 ulp for its own, the table's last
operation and c_0 add at most 1 each, so the two differ by at most 3 ulp."""
import os
import subprocess

import numpy as np
import pytest

from oracle import hopf_pdhg as HO
from oracle import lax_pdhg as O
from oracle import lax_schemes as SO
from paper_1803_01215_gb300 import binding, build_lib, workloads as W

torch = pytest.importorskip("torch")

from gpu_common import gpu  # noqa: E402

pytestmark = pytest.mark.gpu


def _fixed(w, precision, K, **kw):
    return gpu(w, precision, tol=0.0, max_iter=K, check_every=K, **kw)


def _ragged(w, Ns, precision, K):
    """The points of workload w, point b with Ns[b] steps, through a ragged plan."""
    prob = binding.Problem.from_workload(w)
    opts = binding.make_opts(sigma=w["sigma"], tau=w["tau"], tol=0.0, max_iter=K, check_every=K, seed=w["seed"],
                             init_radius=w["init_radius"], precision=precision)
    plan = binding.RaggedPlan([prob], np.zeros(len(Ns), np.int32), np.asarray(Ns, np.int32), opts)
    xq = torch.as_tensor(plan.pack_xq(list(w["xq"])), device="cuda")
    out = plan.solve(xq, torch.as_tensor(w["t"], device="cuda"), return_traj=True)
    return plan, {k: v.cpu().numpy() for k, v in out.items()}


@pytest.mark.parametrize("d,N", [(3, 1), (11, 4), (63, 9), (64, 1), (65, 7), (130, 5), (1030, 3), (1030, 9)])
def test_eikonal_without_node_guards_gives_the_guarded_bits(d, N):
    w = W.eikonal(d=d, sign=-1, t=N * W.EIK_DELTA, B=5, seed=4)
    u = _fixed(w, "fp32", 48)
    plan, r = _ragged(w, [N] * 5, "fp32", 48)
    np.testing.assert_array_equal(u["traj_x"].ravel(), r["traj_x"])
    np.testing.assert_array_equal(u["traj_p"].ravel(), r["traj_p"])
    np.testing.assert_array_equal(u["V"], r["V"])


@pytest.mark.parametrize("d", [5, 12, 32, 37, 64, 65, 100, 104, 105, 128])
def test_tiles_past_the_last_node_leave_the_others_alone(d):
    """A ragged batch runs every N of a class at the class's largest; each point's
    iterates are those of its own uniform launch."""
    Ns = [1, 3, 4, 5, 8, 9, 17, 23, 32] + ([33, 40, 63, 64] if d <= 105 else [])
    w = W.tanh_drift(d, B=len(Ns), seed=6)
    plan, r = _ragged(w, Ns, "fp32", 24)
    for b, N in enumerate(Ns):
        wb = W.subset(w, [b])
        wb["N"] = N
        u = _fixed(wb, "fp32", 24, point_offset=b)
        np.testing.assert_array_equal(u["traj_x"][0], plan.point_traj(r["traj_x"], b))
        np.testing.assert_array_equal(u["traj_p"][0], plan.point_traj(r["traj_p"], b))
        o = O.solve(wb, tol=0.0, max_iter=24, check_every=24)
        assert np.max(np.abs(u["traj_x"][0] - o["x"][0])) <= 1e-4       # 24 steps' FP32 rounding, d terms
        assert np.max(np.abs(u["traj_p"][0] - o["p"][0])) <= 1e-4


@pytest.mark.parametrize("form", ["lax", "hopf", "trap"])
@pytest.mark.parametrize("d,N", [(6, 1), (8, 3), (13, 4), (13, 5), (32, 8), (33, 12), (5, 32)])
def test_fp64_drift_tiles_from_node_one(d, N, form):
    w = W.tanh_drift(d, B=4, seed=8)
    w["N"] = N
    kw = dict(tol=0.0, max_iter=40, check_every=40)
    if form == "trap":
        g, o = _fixed(w, "fp64", 40, scheme="trap"), SO.solve_scheme(w, "trap", **kw)
        np.testing.assert_allclose(g["V"], o["V"], rtol=0, atol=1e-10)
        assert np.max(np.abs(g["traj_x"] - o["x"])) <= 1e-10
        return
    g = _fixed(w, "fp64", 40, formulation=form)
    o = O.solve(w, **kw) if form == "lax" else HO.solve_hopf(w, **kw)
    assert np.max(np.abs(g["traj_x"] - o["x"])) <= 1e-10
    assert np.max(np.abs(g["traj_p"] - o["p"])) <= 1e-10


TANH = r"""
#include <cstdio>
#include "hj_internal.cuh"
#include "tanh64.cuh"
__device__ long long order(double x) {
  const long long b = __double_as_longlong(x);
  return b < 0 ? (long long)0x8000000000000000ull - b : b;
}
__global__ void k(long long* worst, int* bad) {
  extern __shared__ double tab[];
  hj::tanh_taylor_table(tab, threadIdx.x, blockDim.x);
  __syncthreads();
  long long w = 0;
  const long long n = 1ll << 26, step = (long long)gridDim.x * blockDim.x;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += step) {
    // both signs over [-20, 20], and magnitudes from 2^-60 up
    const double u = (double)i / n;
    const double xs[3] = {40.0 * u - 20.0, exp2(70.0 * u - 60.0), -exp2(8.0 * u - 7.0)};
    for (int q = 0; q < 3; ++q) {
      const long long e = llabs(order(hj::tanh_taylor(xs[q], tab)) - order(tanh(xs[q])));
      w = e > w ? e : w;
    }
  }
  atomicMax((unsigned long long*)worst, (unsigned long long)w);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const double inf = __longlong_as_double(0x7ff0000000000000ll), nan = __longlong_as_double(0x7ff8000000000000ll);
    int b = 0;
    b += hj::tanh_taylor(inf, tab) != 1.0;
    b += hj::tanh_taylor(-inf, tab) != -1.0;
    b += hj::tanh_taylor(nan, tab) == hj::tanh_taylor(nan, tab);
    b += hj::tanh_taylor(0.0, tab) != 0.0;
    b += hj::tanh_taylor(1e300, tab) != 1.0;
    *bad = b;
  }
}
int main() {
  long long *w, hw = 0; int *b, hb = 1;
  cudaMalloc(&w, 8); cudaMalloc(&b, 4); cudaMemset(w, 0, 8);
  k<<<304, 256, hj::kTanhRows * hj::kTanhRow * 8>>>(w, b);
  cudaMemcpy(&hw, w, 8, cudaMemcpyDeviceToHost); cudaMemcpy(&hb, b, 4, cudaMemcpyDeviceToHost);
  printf("%lld %d %d\n", hw, hb, (int)cudaDeviceSynchronize());
}
"""


def test_taylor_table_tanh(tmp_path):
    src, exe = tmp_path / "tanh.cu", tmp_path / "tanh"
    src.write_text(TANH)
    subprocess.run([build_lib.nvcc_path(), *build_lib.ARCH, *build_lib.NVCC_FLAGS, str(src), "-o", str(exe)], check=True)
    worst, bad, err = subprocess.run([str(exe)], capture_output=True, text=True, check=True,
                                     env=dict(os.environ)).stdout.split()
    print("tanh: largest distance from CUDA's", worst, "ulp")
    assert int(err) == 0 and int(bad) == 0
    assert int(worst) <= 3


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("d,N", [(1, 1), (3, 15), (4, 16), (5, 17), (37, 33), (64, 40), (100, 5)])
def test_drift_gradient_at_any_trajectory(d, N, precision):
    """hj_solve_grad against the envelope formulas in FP64 at random trajectories: FP64
    sums of B N d products to 1e-12 of their size, FP32 products to 2e-6 of it."""
    rng = np.random.default_rng(d * 100 + N)
    B = 9
    w = W.tanh_drift(d, B=B, seed=2)
    w["N"] = N
    prob = binding.Problem.from_workload(w)
    T = torch.float32 if precision == "fp32" else torch.float64
    X = torch.as_tensor(rng.standard_normal((B, N + 1, d)), device="cuda").to(T)
    P = torch.as_tensor(rng.standard_normal((B, N + 1, d)), device="cuda").to(T)
    t = torch.as_tensor(w["t"], device="cuda")
    wt = torch.as_tensor(rng.uniform(0.5, 1.5, B), device="cuda")
    g = binding.solve_grad(prob, t, N, precision, X, P, wt)
    A = torch.as_tensor(w["dyn"].reshape(d, d), device="cuda")
    x, p, delta = X.double()[:, 1:], P.double()[:, 1:], (t / N)[:, None]
    u = p * (1.0 - torch.tanh(x @ A.T) ** 2)
    dA = -torch.einsum("b,bji,bjk->ik", wt * delta[:, 0], u, x)
    dxq = wt[:, None] * (p[:, -1] - delta * (u[:, -1] @ A))
    e = X.double()[:, 0] - torch.as_tensor(w["c"], device="cuda")
    rt = 1e-12 if precision == "fp64" else 2e-6
    size = float(torch.einsum("b,bji,bjk->ik", wt * delta[:, 0], u.abs(), x.abs()).max())
    assert float((g["ddyn"].reshape(d, d) - dA).abs().max()) <= rt * size
    assert float((g["dxq"] - dxq).abs().max()) <= 10 * rt * max(1.0, float(dxq.abs().max()))
    assert float((g["dc"] + (wt[:, None] * e).sum(0)).abs().max()) <= 10 * rt * B
