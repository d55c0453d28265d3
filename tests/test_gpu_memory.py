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


@pytest.mark.parametrize("precision,tol", [(32, 2e-5), (64, 1e-12)])
def test_instances_of_a_batch_hold_one_grid(precision, tol):
    """A batch's instances are evaluated in the batch's buffers: their plans hold no second grid, until one
    is solved on its own, which gives what the batch gives (sums in another order), call after call."""
    import paper_0807_2387_gb300 as fs
    rng = np.random.default_rng(4)
    dev = torch.device("cuda", 0)
    pts = torch.tensor(rng.uniform(-0.17, 0.17, (3000, 2)), device=dev)
    q = torch.tensor(rng.standard_normal((2, 3000)), device=dev)
    batch = fs.FastSumBatch([(pts, pts, 512, 4 / 512)], 2.0, 4, 2, precision=precision)
    alone = fs.FastSum(pts, pts, 512, 2.0, 4, 4 / 512, precision=precision)
    member = batch.plan(0)
    grid = 512 * 512 * precision // 8
    assert member.info["workspace_bytes"] <= alone.info["workspace_bytes"] - grid
    H = batch.eval([q])[1][0].double()
    for charges, want in ((q[0], H[0]), (q, H), (q[1], H[1])):
        got = member.set_charges(charges).field()[1].double()
        assert float((got - want).norm() / want.norm()) <= tol
    H2 = batch.eval([q])[1][0].double()
    assert float((H2 - H).norm() / H.norm()) <= tol
    for plan in (member, alone, batch):
        plan.close()
