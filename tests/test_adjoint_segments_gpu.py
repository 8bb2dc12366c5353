"""The reverse sweep's segments: the gradient does not depend on the checkpoint
spacing.  Each iteration's transposed step reads the same values whatever the
segment it falls in, so dV/dx_q is the same to the bit and the sums over
iterations differ by their order alone: at most K (a few hundred) rounded
additions of 2^-53, below 1e-12 of the sums' largest term."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_01215_gb300 import binding, workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


def _grad(w, precision, C, cap=None):
    prob = binding.Problem.from_workload(w)
    opts = binding.make_opts(sigma=w["sigma"], tau=w["tau"], tol=0.0, max_iter=w["max_iter"], check_every=1,
                             seed=w["seed"], init_radius=w["init_radius"], precision=precision)
    xq = torch.as_tensor(w["xq"], device="cuda")
    t = torch.as_tensor(w["t"], device="cuda")
    iters = torch.as_tensor(w["iters"], dtype=torch.int32, device="cuda")
    weight = torch.linspace(0.5, 1.5, len(xq), dtype=torch.float64, device="cuda")
    g = binding.solve_grad_unrolled(prob, xq, t, int(w["N"]), opts, iters, weight, checkpoint_every=C, max_iters=cap)
    return {k: v.cpu().numpy() for k, v in g.items()}


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("family,N", [("quadcopter", 1), ("quadcopter", 32), ("quadcopter", 33), ("quadcopter", 65),
                                      ("quadratic", 20), ("quadratic", 64)])
def test_gradient_is_independent_of_the_spacing(family, N, precision):
    w = W.quadcopter(B=5, seed=3, N=N, t=0.4) if family == "quadcopter" else W.quadratic_closed_form(B=5)
    w["N"] = N
    # iteration counts at the segments' edges: none, one, a whole segment, one more, several
    w["iters"] = np.array([0, 1, 64, 65, 131])
    base = _grad(w, precision, 1)
    assert np.all(np.isfinite(base["dxq"]))
    for C in (7, 64, 65, 1000):
        g = _grad(w, precision, C, cap=131 if C < 65 else 200)
        np.testing.assert_array_equal(g["dxq"], base["dxq"])
        for k in ("dW", "dc", "ddyn"):
            np.testing.assert_allclose(g[k], base[k], rtol=0, atol=1e-11 * max(1.0, np.max(np.abs(base[k]), initial=0.0)))
