"""Accuracy of several charge vectors of one plan, evaluated together (GPU)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nrhs", [2, 3, 4])
@pytest.mark.parametrize("lines", [4, 6])
def test_vectors_together_are_as_accurate_as_alone(nrhs, lines):
    """A crowded cell, 12,000 charges of one sign within reach of every target: the RMS error of FP32 sums
    against FP64 with `nrhs` copies of the vector in one call is at most 1.5 times that of the vector alone.
    The pair arithmetic is the same or, of the two forms of the gradient's coefficient, the more exact one; the
    sums' order and the grid's atomics change the rest by a few per cent.  (One running FP32 sum over the
    candidates in place of partial sums per list multiplies the errors by two to five.)"""
    import paper_0807_2387_gb300 as fs
    rng = np.random.default_rng(10 * nrhs + lines)
    rim = 0.24 * np.stack([np.cos(np.arange(5)), np.sin(np.arange(5))], 1)
    src = np.concatenate([rng.uniform(0.002, 0.030, (12000, 2)), rim])
    tgt = np.concatenate([rng.uniform(0.002, 0.030, (6000, 2)), -rim])
    dev = torch.device("cuda", 0)
    s, t = torch.tensor(src, device=dev), torch.tensor(tgt, device=dev)
    q = torch.tensor(rng.uniform(0.5, 1.5, len(src)).astype(np.float32), device=dev)

    def field(precision, charges):
        plan = fs.FastSum(s, t, 32, 2.0, 5, lines / 32, precision=precision)
        return [v.double() for v in plan.set_charges(charges).field(dtype=torch.float64)]

    ref, alone, together = field(64, q), field(32, q), field(32, q.repeat(nrhs, 1))
    for name, r, a, b in zip(("phi", "H"), ref, alone, together):
        rms = float((a - r).square().mean().sqrt())
        for k in range(nrhs):
            got = float((b[k] - r).square().mean().sqrt())
            assert got <= 1.5 * rms, (name, k, got, rms)
