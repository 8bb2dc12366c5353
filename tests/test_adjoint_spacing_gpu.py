"""Checkpoints as far apart as the caller asks for.  dV/dx_q does not depend on the
spacing to the bit; the sums over iterations by their order alone: fewer than 500 rounded
additions of 2^-53, below 1e-12 of the sums' largest term."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_01215_gb300 import binding, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _grad(w, precision, C, cap):
    prob = binding.Problem.from_workload(w)
    opts = binding.make_opts(sigma=w["sigma"], tau=w["tau"], tol=0.0, max_iter=w["max_iter"], check_every=1,
                             seed=w["seed"], init_radius=w["init_radius"], precision=precision)
    xq = torch.as_tensor(w["xq"], device="cuda")
    t = torch.as_tensor(w["t"], device="cuda")
    iters = torch.as_tensor(w["iters"], dtype=torch.int32, device="cuda")
    weight = torch.linspace(0.5, 1.5, len(xq), dtype=torch.float64, device="cuda")
    g = binding.solve_grad_unrolled(prob, xq, t, int(w["N"]), opts, iters, weight, checkpoint_every=C, max_iters=cap)
    return {k: v.cpu().numpy() for k, v in g.items()}


def _same(g, base):
    np.testing.assert_array_equal(g["dxq"], base["dxq"])
    for k in ("dW", "dc", "ddyn"):
        np.testing.assert_allclose(g[k], base[k], rtol=0, atol=1e-11 * max(1.0, np.max(np.abs(base[k]), initial=0.0)))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("family,N", [("quadcopter", 40), ("quadratic", 20)])
def test_long_segments(family, N, precision):
    w = W.quadcopter(B=12, seed=3, N=N, t=0.4) if family == "quadcopter" else W.quadratic_closed_form(B=12)
    w["N"] = N
    # at the edges of a 64-step piece, of a segment of 130 and of several of both
    w["iters"] = np.array([0, 1, 63, 64, 65, 128, 129, 130, 131, 260, 261, 400])
    base = _grad(w, precision, 1, 400)
    assert np.all(np.isfinite(base["dxq"]))
    for C, cap in [(65, 400), (128, 401), (129, 400), (130, 400), (200, 400), (400, 400), (1000, 400), (5000, 10**6)]:
        _same(_grad(w, precision, C, cap), base)


def test_spacing_bounds_the_workspace():
    """2e9 iterations at most, checkpoints every 1e6: 2001 checkpoints (37 MB per CTA) and the
    pieces of one segment.  At one checkpoint per 64 iterations a single CTA would need 580 GB."""
    w = W.quadcopter(B=3, seed=3, N=128, t=0.4)
    w["iters"] = np.array([5, 70, 140])
    _same(_grad(w, "fp32", 1_000_000, 2_000_000_000), _grad(w, "fp32", 1, 140))


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_pieces_longer_than_64_steps(precision):
    """Checkpoints every 1e6 iterations: pieces of 1000 steps, the parameter sums folded every 64."""
    w = W.quadcopter(B=4, seed=3, N=20, t=0.4)
    w["iters"] = np.array([64, 65, 700, 1001])
    _same(_grad(w, precision, 1_000_000, 1_000_000), _grad(w, precision, 1, 1001))
