"""Device memory that plans hold (GPU)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("precision", [32, 64])
def test_growing_number_of_charge_vectors(precision):
    """A plan used with 1, 2, 3 and then 4 charge vectors holds what one used with 4 at once holds: buffers
    outgrown are given back.  A set of buffers of one vector is 17 MB and more here, the allocator's
    rounding below 8 MB in all."""
    import paper_0807_2387_gb300 as fs
    rng = np.random.default_rng(3)
    dev = torch.device("cuda", 0)
    pts = torch.tensor(rng.uniform(-0.17, 0.17, (300000, 2)), device=dev)
    q = torch.tensor(rng.standard_normal((4, 300000)), device=dev)
    held, out = {}, {}
    for name, counts in (("warm", (4,)), ("at once", (4,)), ("growing", (1, 2, 3, 4))):
        plan = fs.FastSum(pts, pts, 1024, 2.0, 4, 4 / 1024, precision=precision)
        before = _free()
        for r in counts:
            plan.set_charges(q[:r])
        held[name] = before - _free()
        out[name] = plan.field()[1].double()
        plan.sync()
        plan.close()
    assert held["growing"] <= held["at once"] + 8 * 2 ** 20, held
    err = float((out["growing"] - out["at once"]).norm() / out["at once"].norm())
    assert err <= (1e-12 if precision == 64 else 2e-5), err
