"""The register-tiled drift kernel's two instantiations (the Lax form with theta = 1, and
the one that takes the form and theta from the options) run the same arithmetic.

theta enters z^1 only, and z^1 the second iteration only; the Hopf form differs from the
Lax form at x_0 and in node 1's prox.  After one iteration from the same guess the FP32
iterates are therefore the same bits: all of them for any theta, those of the nodes from
the second on for the Hopf form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_01215_gb300 import workloads as W  # noqa: E402

from gpu_common import gpu  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N", [(13, 7), (13, 33), (32, 8), (32, 32), (37, 24), (64, 5), (64, 100), (65, 32), (100, 16),
                                 (128, 40)])
def test_first_iteration_is_the_same_in_every_form(d, N):
    w = W.tanh_drift(d, B=6, seed=5, N=N)
    kw = dict(tol=0.0, max_iter=1, check_every=1)
    base = gpu(w, "fp32", **kw)
    for theta in (0.5, 0.0):
        g = gpu(w, "fp32", theta=theta, **kw)
        np.testing.assert_array_equal(g["traj_p"], base["traj_p"])
        np.testing.assert_array_equal(g["traj_x"], base["traj_x"])
    h = gpu(w, "fp32", formulation="hopf", **kw)
    np.testing.assert_array_equal(h["traj_p"][:, 2:], base["traj_p"][:, 2:])
    np.testing.assert_array_equal(h["traj_x"][:, 2:], base["traj_x"][:, 2:])
