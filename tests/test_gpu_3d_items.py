"""FP32 3D plans whose points make unusual items, against FP64 within the bar of the 3D gates (GPU)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def rel(a, b):
    return max(float((a - b).norm() / b.norm()), float((a - b).abs().max() / b.abs().max()))


def _fields(src, tgt, q, n, m, eps, **opts):
    import paper_0807_2387_gb300 as fs
    dev = torch.device("cuda", 0)
    out = {}
    for precision in (64, 32):
        plan = fs.FastSum3(*(torch.tensor(v, device=dev) for v in (src, tgt)), n, 2.0, m, eps, precision=precision, **opts)
        out[precision] = plan.set_charges(torch.tensor(q, device=dev)).field(dtype=torch.float64)
        plan.sync()
        info = plan.info
        plan.close()
    return out[32], out[64], info


@pytest.mark.parametrize("m", [2, 4])
def test_3d_crowds_at_the_ends_of_the_domain(m):
    """Cells of several items each at the six ends of the axes, where a point's taps reach the last lines of
    the active window."""
    rng = np.random.default_rng(m)
    ends = 0.25 * np.concatenate([np.eye(3), -np.eye(3)])
    src = np.concatenate([ends, (ends[:, None] * (1 - 10.0 ** rng.uniform(-4, -2, (6, 150, 1)))).reshape(-1, 3)])
    got, want, _ = _fields(src, src[::-1] * 1.0, rng.standard_normal(len(src)), 32, m, 3 / 32)
    assert rel(got[0], want[0]) <= 5e-6 and rel(got[1], want[1]) <= 5e-6, (rel(got[0], want[0]), rel(got[1], want[1]))


@pytest.mark.parametrize("m", [2, 3, 5])
@pytest.mark.parametrize("ns,nt", [(2500, 1900), (9000, 1300)])
def test_3d_fp32_every_width(m, ns, nt):
    """Window widths other than the default's, targets and sources as the near field's items."""
    rng = np.random.default_rng(m + ns)
    src, tgt = (rng.uniform(-0.14, 0.14, (k, 3)) for k in (ns, nt))
    tgt[:200] = src[:200]
    got, want, _ = _fields(src, tgt, rng.standard_normal(ns), 32, m, 3 / 32)
    assert rel(got[0], want[0]) <= 5e-6 and rel(got[1], want[1]) <= 5e-6, (rel(got[0], want[0]), rel(got[1], want[1]))


@pytest.mark.parametrize("n,nt", [(128, 300000), (256, 800000)])
def test_3d_crowded_cell_among_sparse_ones(n, nt):
    """A cell of more targets than one sorted run holds (2,048), where the mean over all targets makes
    items of 16 and of 8."""
    rng = np.random.default_rng(n)
    v = rng.standard_normal((nt, 3))
    tgt = 0.25 * rng.random((nt, 1)) ** (1 / 3) * v / np.linalg.norm(v, axis=1)[:, None]
    eps = 1 / n
    tgt[-1] = [0.0, 0.0, 0.25]                                      # the scale is known
    scale, n_os = (0.25 - eps / 2) / 0.25, 2 * n
    lo = int(np.floor(n_os * (0.25 + 0.5 * eps))) - 5               # the window's first line; cells of two lines
    centre = (lo + 2 * np.array([n // 3, n // 4, n // 3 + 2]) + 1) / n_os - 0.5
    crowd = centre / scale + rng.uniform(-1e-4, 1e-4, (2100, 3))
    tgt[:2100] = crowd
    src = np.concatenate([crowd[:300] + rng.uniform(-1e-4, 1e-4, (300, 3)), tgt[5000:8000]])
    got, want, info = _fields(src, tgt, rng.standard_normal(len(src)), n, 4, eps, p=2)
    assert (info["window_lo"], info["cell"]) == (lo, 2) and abs(info["scale"] - scale) < 1e-12
    line = np.floor(info["n_os"] * (info["scale"] * crowd)) + info["n_os"] // 2 - info["window_lo"]
    assert len(np.unique(line // info["cell"], axis=0)) == 1        # one cell
    key = np.floor(info["n_os"] * (info["scale"] * tgt)) + info["n_os"] // 2 - info["window_lo"]
    _, counts = np.unique(key // info["cell"], axis=0, return_counts=True)
    mean = (counts.astype(float) ** 2).sum() / nt
    assert (8 <= mean < 20) if n == 128 else mean < 8, mean
    assert rel(got[0], want[0]) <= 5e-6 and rel(got[1], want[1]) <= 5e-6, (rel(got[0], want[0]), rel(got[1], want[1]))
