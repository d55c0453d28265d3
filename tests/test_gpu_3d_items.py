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
