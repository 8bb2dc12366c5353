"""FP32 parameter sums of the reverse sweep beyond FP32's range.  Every term of the a_h sum
is an FP32 number below 3.4e38 here and their sum is above: as an FP64 sum it is finite.

One step, one node, no thrust and no gravity: the a_h gradient is - sum_r L w_r a_r with
w = - 3/4 c on rows 6 and 7 (x_1 = 0, x_0 = c / 2 by tau W^2 = 1, and x_0's own adjoint),
a = (1, 1, 0) / sqrt 2 and L = 1e22."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1803_01215_gb300 import binding  # noqa: E402

pytestmark = pytest.mark.gpu


def _ddyn(precision):
    sigma, t = 1e19, 1000.0
    tau = 0.2 / sigma
    W, c, x = np.ones(12), np.zeros(12), np.zeros(12)
    W[6:8] = np.sqrt(1.0 / tau)
    c[6:8] = 2.9e38 / (sigma * t) / 0.75
    x[3], x[4] = np.pi / 4, np.pi / 2
    prob = binding.Problem("quadcopter", 12, np.array([1e20, 0.0, 0.0, 0.0]), W, c)
    opts = binding.make_opts(sigma=sigma, tau=tau, tol=0.0, max_iter=1, check_every=1, seed=1, init_radius=1e-22,
                             precision=precision)
    dev = dict(device="cuda", dtype=torch.float64)
    g = binding.solve_grad_unrolled(prob, torch.as_tensor(x[None], **dev), torch.full((1,), t, **dev), 1, opts,
                                    torch.ones(1, dtype=torch.int32, device="cuda"), torch.ones(1, **dev))
    return g["ddyn"].cpu().numpy()


def test_sum_beyond_the_range_of_fp32():
    f64, f32 = _ddyn("fp64"), _ddyn("fp32")
    expect = 2.9e38 * np.sqrt(2.0)
    assert abs(f64[1] / expect - 1.0) <= 1e-6
    assert abs(f32[1] / expect - 1.0) <= 1e-5        # a handful of FP32 roundings
