"""FP64 drift kernel with several points per CTA (more points than SMs): each point gives
the bits that it gives in a batch small enough for one point per CTA, and those are the
oracle's to 1e-10 after 24 iterations."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import hopf_pdhg as HO  # noqa: E402
from oracle import lax_pdhg as O  # noqa: E402
from oracle import lax_schemes as SO  # noqa: E402
from paper_1803_01215_gb300 import binding, workloads as W  # noqa: E402

from gpu_common import gpu  # noqa: E402

pytestmark = pytest.mark.gpu

K = 24
KW = dict(tol=0.0, max_iter=K, check_every=K)
CHUNK = 100


def _batch():
    return 2 * torch.cuda.get_device_properties(0).multi_processor_count + 97


@pytest.mark.parametrize("form", ["lax", "hopf", "trap"])
@pytest.mark.parametrize("d,N", [(32, 32), (33, 30), (64, 24)])
def test_points_of_a_shared_cta(d, N, form):
    B = _batch()
    w = W.tanh_drift(d, B=B, seed=7, N=N)
    kw = dict(KW, scheme="trap") if form == "trap" else dict(KW, formulation=form)
    g = gpu(w, "fp64", **kw)
    for b0 in range(0, B, CHUNK):
        part = gpu(W.subset(w, range(b0, min(b0 + CHUNK, B))), "fp64", point_offset=b0, **kw)
        for k in ("traj_x", "traj_p", "V"):
            np.testing.assert_array_equal(g[k][b0:b0 + CHUNK], part[k])
    ids = [0, 1, B // 2, B - 1]
    s = W.subset(w, ids)
    o = SO.solve_scheme(s, "trap", **KW) if form == "trap" else (O.solve(s, **KW) if form == "lax" else HO.solve_hopf(s, **KW))
    assert np.max(np.abs(g["traj_x"][ids] - o["x"])) <= 1e-10
    p = g["traj_p"][ids, 1:] if form == "trap" else g["traj_p"][ids]    # that oracle's p: nodes 1..N
    assert np.max(np.abs(p - o["p"])) <= 1e-10


def _plan(w, Ns, b0=0):
    prob = binding.Problem.from_workload(w)
    opts = binding.make_opts(sigma=w["sigma"], tau=w["tau"], seed=w["seed"], init_radius=w["init_radius"], precision="fp64",
                             point_offset=b0, **KW)
    plan = binding.RaggedPlan([prob], np.zeros(len(Ns), np.int32), np.asarray(Ns, np.int32), opts)
    xq = torch.as_tensor(plan.pack_xq(list(w["xq"])), device="cuda")
    out = plan.solve(xq, torch.as_tensor(w["t"], device="cuda"), return_traj=True)
    return plan, {k: v.cpu().numpy() for k, v in out.items()}


def test_points_of_a_shared_cta_with_their_own_node_counts():
    B = _batch()
    w = W.tanh_drift(32, B=B, seed=9)
    Ns = [(32, 31, 24, 21, 4, 1, 30)[b % 7] for b in range(B)]      # whole tiles and not, in one bucket
    plan, r = _plan(w, Ns)
    for b0 in range(0, B, CHUNK):
        n = min(CHUNK, B - b0)
        sub, s = _plan(W.subset(w, range(b0, b0 + n)), Ns[b0:b0 + n], b0)
        for i in range(n):
            np.testing.assert_array_equal(plan.point_traj(r["traj_x"], b0 + i), sub.point_traj(s["traj_x"], i))
            np.testing.assert_array_equal(plan.point_traj(r["traj_p"], b0 + i), sub.point_traj(s["traj_p"], i))
        np.testing.assert_array_equal(r["V"][b0:b0 + n], s["V"])
    for b in (0, 1, 4, 5, B - 1):
        wb = W.subset(w, [b])
        wb["N"] = Ns[b]
        o = O.solve(wb, **KW)
        assert np.max(np.abs(plan.point_traj(r["traj_x"], b) - o["x"][0])) <= 1e-10
