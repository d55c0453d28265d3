"""Pairs much closer than eps_I: the near field at distances that only some places of the domain can hold
(GPU).

Doubles are finest near the coordinate origin, so distinct points there may be any distance apart.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

#: distances from the source at the origin, in the caller's units
TINY = np.array([1e-17, 1e-19, 3e-20, 1e-20, 1e-21, 1e-22, 1e-30, 1e-45, 1e-60])


def _around_the_origin(seed):
    """A unit source at the origin, targets at TINY from it, and some ordinary points of both kinds."""
    rng = np.random.default_rng(seed)
    t = rng.uniform(0.0, 2.0 * np.pi, len(TINY))
    near = TINY[:, None] * np.stack([np.cos(t), np.sin(t)], 1)
    src = np.concatenate([[[0.0, 0.0]], rng.uniform(-0.17, 0.17, (60, 2)), [[0.25, 0.0]]])
    tgt = np.concatenate([near, rng.uniform(-0.17, 0.17, (40, 2))])
    return src, tgt, np.concatenate([[1.0], rng.standard_normal(len(src) - 1)])


@pytest.mark.parametrize("p", [1, 2, 4])
def test_fp64_log_of_very_close_pairs(p):
    """phi, H and dL/dq of FP64 plans and phi of an FP64 batch at the targets a tiny distance from a
    source, each within 1e-12 of the oracle's (the bar of the FP64 gates), element by element: phi grows
    with the logarithm of the distance and H with its inverse.  (m = 8: the origin is a grid line, where the
    narrower windows' edge values, 1e-9 of the peak at m = 5, are added or not by the last bit.)"""
    import paper_0807_2387_gb300 as fs
    from oracle import fastsum as F
    from oracle import kernel as K
    src, tgt, q = _around_the_origin(p)
    eps, k = 4 / 64, len(TINY)
    par = K.make_params(64, 2.0, 8, eps, p)
    phi_o, H_o = F.fast_sum(src, tgt, q, par, "nfft")
    dev = torch.device("cuda", 0)
    s, t, qd = (torch.tensor(v, device=dev) for v in (src, tgt, q))
    plan = fs.FastSum(s, t, 64, 2.0, 8, eps, precision=64, p=p)
    phi, H = (v.cpu().numpy() for v in plan.set_charges(qd).field())
    assert np.max(np.abs(phi - phi_o) / np.abs(phi_o).clip(0.1)) <= 1e-12
    assert np.max(np.linalg.norm((H - H_o)[:k], axis=1) / np.linalg.norm(H_o[:k], axis=1)) <= 1e-12
    batch = fs.FastSumBatch([(s, t, 64, eps)], 2.0, 8, 1, precision=64, p=p)
    phi_b = batch.eval([qd[None]])[0][0].cpu().numpy().reshape(-1)
    assert np.max(np.abs(phi_b - phi_o) / np.abs(phi_o).clip(0.1)) <= 1e-12
    # dL/dq_0 for dL/dphi = 1 at one target is phi of a unit charge at the origin there
    one = np.zeros(len(src))
    one[0] = 1.0
    unit, _ = F.fast_sum(src, tgt, one, par, "nfft")
    for i in range(k):
        g = torch.zeros(len(tgt), dtype=torch.float64, device=dev)
        g[i] = 1.0
        dq = plan.adjoint(g, None, want_q=True)[0]
        assert abs(float(dq[0]) - unit[i]) <= 1e-12 * abs(unit[i]), (TINY[i], float(dq[0]), unit[i])


@pytest.mark.parametrize("m", [2, 3, 4, 5])
def test_fp64_points_just_below_a_grid_line(m):
    """FP64 plans with coordinates a negative fraction of the last place from 0, a grid line: the fraction
    to the line below rounds to 1, and the first tap then lies on the window's (open) edge, where it counts
    nothing.  Field, gradients and Hessian against the oracle within 1e-12, the bar of the FP64 gates; the
    edge's closed value is 1e-3 (m = 2) to 1e-9 (m = 5) of the peak."""
    import paper_0807_2387_gb300 as fs
    from oracle import adjoint as A
    from oracle import fastsum as F
    from oracle import kernel as K
    rng = np.random.default_rng(m)
    src, tgt = (rng.uniform(-0.17, 0.17, (k, 2)) for k in (60, 50))
    for pts in (src, tgt):
        pts[:10, 0] = -1e-22 * rng.uniform(1.0, 9.0, 10)
        pts[10:20, 1] = -1e-25 * rng.uniform(1.0, 9.0, 10)
    src, tgt = np.concatenate([src, [[0.25, 0.0]]]), np.concatenate([tgt, [[0.0, 0.25]]])
    q, gp, gh = rng.standard_normal(len(src)), rng.standard_normal(len(tgt)), rng.standard_normal((len(tgt), 2))
    par = K.make_params(64, 2.0, m, 4 / 64)
    dev = torch.device("cuda", 0)
    s, t, qd, gpd, ghd = (torch.tensor(v, device=dev) for v in (src, tgt, q, gp, gh))
    plan = fs.FastSum(s, t, 64, 2.0, m, 4 / 64, precision=64)
    got = (*plan.set_charges(qd).field(), *plan.adjoint(gpd, ghd, True, True, True))
    want = (*F.fast_sum(src, tgt, q, par, "nfft"), *A.fast_sum_adjoint(src, tgt, q, gp, gh, par))
    for name, a, b in zip(("phi", "H", "dq", "dsrc", "dtgt"), got, want):
        a = a.cpu().numpy()
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b)), (name, np.max(np.abs(a - b)) / np.max(np.abs(b)))


#: distances of FP32 3D pairs in torus units: above the FP32 kernels' floor of w (1e-10 eps_I), and below it
CLOSE3 = 10.0 ** np.linspace(-10.3, -5.0, 22)
TOUCHING3 = np.array([1e-15, 3e-16, 1e-16])


@pytest.mark.parametrize("source_major", [False, True])
def test_3d_fp32_close_pairs(source_major):
    """3D FP32 plans, point pairs at CLOSE3: phi and H of each target (its pair dominates them) against the
    FP64 plan within 5e-6, the bar of the 3D gates.  Pairs at TOUCHING3 are a few units in the last place
    apart, distinct all the same: not taken for coincident ones, whose charge is left out (phi at least
    that of a pair at the floor of w)."""
    import paper_0807_2387_gb300 as fs
    rng = np.random.default_rng(7 + source_major)
    n, eps = 32, 4 / 32
    scale = (0.25 - eps / 2) / 0.25          # of caller's units to torus units; the rim below fixes it
    dist = np.concatenate([np.repeat(CLOSE3, 8), np.repeat(TOUCHING3, 40)])
    d = rng.standard_normal((len(dist), 3))
    d *= (dist / scale / np.linalg.norm(d, axis=1))[:, None]
    # the pairs lie eps_I / 4 and more from each other, a charge of 1 each, the rest a thousandth
    g = np.stack(np.meshgrid(*[np.linspace(-0.13, 0.13, 9)] * 3, indexing="ij"), -1).reshape(-1, 3)
    at = g[rng.permutation(len(g))[: len(dist)]] + rng.uniform(-0.003, 0.003, (len(dist), 3))
    tgt = at + d
    rim = 0.25 * np.concatenate([np.eye(3), -np.eye(3)])
    more = rng.uniform(-0.12, 0.12, (4 * len(tgt) if source_major else 40, 3))
    src = np.concatenate([at, rim, more])
    q = np.concatenate([np.ones(len(at)), np.zeros(len(rim)), 1e-3 * rng.standard_normal(len(more))])
    keep = np.any(tgt != at, axis=1)         # a difference below the last place would be no difference
    assert keep[: 8 * len(CLOSE3)].all() and keep.mean() > 0.8
    dev = torch.device("cuda", 0)
    s, t, qd = (torch.tensor(v, device=dev) for v in (src, tgt, q))
    got = {}
    for precision in (64, 32):
        plan = fs.FastSum3(s, t, n, 2.0, 4, eps, precision=precision, p=3)
        got[precision] = [v.cpu().numpy() for v in plan.set_charges(qd).field(dtype=torch.float64)]
        plan.sync()
        factor = plan.info["scale"]
    assert abs(factor - scale) < 1e-6
    k = 8 * len(CLOSE3)
    (phi, H), (phi0, H0) = got[32], got[64]
    e_phi, e_h = np.abs(phi - phi0)[:k] / phi0[:k], np.linalg.norm(H - H0, axis=1)[:k] / np.linalg.norm(H0, axis=1)[:k]
    assert e_phi.max() <= 5e-6, (e_phi.max(), dist[e_phi.argmax()])
    assert e_h.max() <= 5e-6, (e_h.max(), dist[e_h.argmax()])
    floor = factor / (4 * np.pi * 1e-10 * eps)
    assert (phi[k:][keep[k:]] >= 0.99 * floor).all(), (phi[k:][keep[k:]].min(), floor)
    assert (phi[k:][~keep[k:]] < 1e-3 * floor).all()
