"""The FP32 near field's items: cells sorted into pieces, 8, 16 or 32 points to a warp (GPU).

The FP64 path, which loops over the points of the cells, is the reference.  Tolerance: 2e-5, the bar of
the FP32-vs-FP64 gates of small cases (FP32 rounding of the pair sums and of the grid, ~1e-6 here).
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def rel(a, b):
    a, b = a.double().cpu().numpy(), b.double().cpu().numpy()
    return max(np.linalg.norm(a - b) / np.linalg.norm(b), np.max(np.abs(a - b)) / np.max(np.abs(b)))


@pytest.mark.parametrize("n_src,n_tgt", [(1, 1), (7, 9), (24, 26), (33, 31), (65, 63), (99, 101), (129, 513), (2048, 2049),
                                         (4500, 40)])
def test_one_crowded_cell(n_src, n_tgt):
    """All points but a rim in one near-field cell: edges of an item (8, 16, 32), of the strips, of a
    sorted run (2048) and of the candidate lists; forward, gradients and Hessian."""
    import paper_0807_2387_gb300 as fs
    rng = np.random.default_rng(n_src + 7 * n_tgt)
    rim = 0.24 * np.stack([np.cos(np.arange(5)), np.sin(np.arange(5))], 1)
    src = np.concatenate([rng.uniform(0.002, 0.030, (n_src, 2)), rim])
    tgt = np.concatenate([rng.uniform(0.002, 0.030, (n_tgt, 2)), -rim])
    dev = torch.device("cuda", 0)
    s, t = torch.tensor(src, device=dev), torch.tensor(tgt, device=dev)
    q = torch.tensor(rng.standard_normal(len(src)), device=dev)
    gp, gh = torch.tensor(rng.standard_normal(len(tgt)), device=dev), torch.tensor(rng.standard_normal((len(tgt), 2)), device=dev)
    got = {}
    for precision in (64, 32):
        plan = fs.FastSum(s, t, 32, 2.0, 5, 4 / 32, precision=precision)
        plan.set_charges(q)
        phi, H = plan.field(dtype=torch.float64)
        got[precision] = (phi, H, *plan.adjoint(gp, gh, True, True, True, dtype=torch.float64))
        plan.sync()
    for name, a, b in zip(("phi", "H", "dq", "dsrc", "dtgt"), got[32], got[64]):
        assert rel(a, b) <= 2e-5, (name, rel(a, b))


@pytest.mark.parametrize("p", [1, 2, 3, 4, 7, 8])
def test_fp64_pair_functions_by_degree(p):
    """The FP64 near field's log, reciprocal and polynomials at every form of the degree, over pairs from
    coincident to eps_I apart: 1e-12 of the oracle, the bar of the FP64 gates."""
    import paper_0807_2387_gb300 as fs
    from oracle import fastsum as F
    from oracle import kernel as K
    rng = np.random.default_rng(90 + p)
    src = rng.uniform(-0.17, 0.17, (333, 2))
    near = src[:200] + 10.0 ** rng.uniform(-9, -1.2, (200, 1)) * rng.standard_normal((200, 2))
    tgt = np.clip(np.concatenate([near, src[200:260], rng.uniform(-0.17, 0.17, (41, 2))]), -0.17, 0.17)
    q = rng.standard_normal(len(src))
    dev = torch.device("cuda", 0)
    plan = fs.FastSum(torch.tensor(src, device=dev), torch.tensor(tgt, device=dev), 64, 2.0, 5, 5 / 64, precision=64, p=p)
    phi, H = plan.set_charges(torch.tensor(q, device=dev)).field()
    phi_o, H_o = F.fast_sum(src, tgt, q, K.make_params(64, 2.0, 5, 5 / 64, p), "nfft")
    for name, a, b in (("phi", phi, phi_o), ("H", H, H_o)):
        assert rel(a, torch.tensor(b)) <= 1e-12, (name, rel(a, torch.tensor(b)))


@pytest.mark.parametrize("nrhs", [2, 3, 4, 5, 9])
@pytest.mark.parametrize("precision,fem", [(32, False), (64, False), (32, True)])
def test_charge_vectors_together(nrhs, precision, fem):
    """Several charge vectors (groups of four and the remainders) against one at a time, which differ by the
    rounding order alone: the FP32-vs-FP64 bar of small cases for FP32, 1e-12 for FP64."""
    import paper_0807_2387_gb300 as fs
    rng = np.random.default_rng(nrhs)
    dev = torch.device("cuda", 0)
    n_src, n_tgt = (3000, 700) if fem else (1500, 1301)      # FEM-like: the near field runs over source items
    s, t = (torch.tensor(rng.uniform(-0.17, 0.17, (k, 2)), device=dev) for k in (n_src, n_tgt))
    q = torch.tensor(rng.standard_normal((nrhs, n_src)), device=dev)
    plan = fs.FastSum(s, t, 64, 2.0, 5, 4 / 64, precision=precision)
    phi, H = plan.set_charges(q).field(dtype=torch.float64)
    tol = 1e-12 if precision == 64 else 2e-5
    for r in range(nrhs):
        one = fs.FastSum(s, t, 64, 2.0, 5, 4 / 64, precision=precision)
        phi1, H1 = one.set_charges(q[r].contiguous()).field(dtype=torch.float64)
        assert rel(phi[r], phi1) <= tol and rel(H[r], H1) <= tol, (r, rel(phi[r], phi1), rel(H[r], H1))
    phi0, H0 = plan.set_charges(q[0].contiguous()).field(dtype=torch.float64)
    assert rel(phi0, phi[0]) <= tol and rel(H0, H[0]) <= tol


@pytest.mark.parametrize("ns,n,lines", [(18000, 64, 2), (15000, 64, 3), (120000, 64, 2), (120000, 64, 4.4)])
def test_3d_run_spreading(ns, n, lines):
    """3D spreading with the sources of a cell in runs of equal base lines: few and many to a run, items of
    one and several pieces, cells of 4, 6 and 9 lines (the widest tile), against FP64 within the FP32
    bar of the 3D gates."""
    import paper_0807_2387_gb300 as fs
    rng = np.random.default_rng(ns)
    v = rng.standard_normal((ns, 3))
    src = 0.25 * v / np.linalg.norm(v, axis=1)[:, None] * rng.random((ns, 1)) ** (1 / 3)
    src[: ns // 4] = src[0] + rng.uniform(-0.004, 0.004, (ns // 4, 3)) if np.linalg.norm(src[0]) < 0.24 else src[: ns // 4]
    dev = torch.device("cuda", 0)
    s, t = torch.tensor(src, device=dev), torch.tensor(src[::3] * 0.97 + 1e-3, device=dev)
    q = torch.tensor(rng.standard_normal(ns), device=dev)
    got = {}
    for precision in (64, 32):
        plan = fs.FastSum3(s, t, n, 2.0, 4, lines / n, precision=precision, p=3)
        got[precision] = plan.set_charges(q).field(dtype=torch.float64)
        plan.sync()
    assert plan.info["spread_items"] > 0
    assert rel(got[32][0], got[64][0]) <= 5e-6, rel(got[32][0], got[64][0])
    assert rel(got[32][1], got[64][1]) <= 5e-6, rel(got[32][1], got[64][1])


@pytest.mark.parametrize("precision,tol", [(32, 2e-5), (64, 1e-12)])
@pytest.mark.parametrize("n", [64, 128])
def test_grid_is_left_clean(n, precision, tol):
    """Every evaluation starts from a zero grid: the same charges give the same field again after other
    charge vectors, several at once, and an adjoint (transform lengths 128 and 256; the sums differ by the
    order of the grid's atomic additions, within the bars of the parity gates)."""
    import paper_0807_2387_gb300 as pkg
    rng = np.random.default_rng(8)
    dev = torch.device("cuda", 0)
    pts = [torch.tensor(rng.uniform(-0.17, 0.17, (k, 2)), device=dev) for k in (700, 500)]
    q = torch.tensor(rng.standard_normal((4, 700)), device=dev)
    fs = pkg.FastSum(*pts, n, 2.0, 4, 4.0 / n, precision=precision)
    first = fs.set_charges(q[0]).field(dtype=torch.float64)
    g = torch.tensor(rng.standard_normal(500), device=dev)
    for again in (lambda: fs.set_charges(q[1]).potential(), lambda: fs.set_charges(q[1:]).field(),
                  lambda: fs.set_charges(q[2]).adjoint(g_phi=g)):
        again()
        for a, b in zip(fs.set_charges(q[0]).field(dtype=torch.float64), first):
            assert float((a - b).norm() / b.norm()) <= tol
    fs.close()


@pytest.mark.parametrize("precision,tol", [(32, 2e-5), (64, 1e-12)])
def test_batch_of_every_line_length(precision, tol):
    """Transform lengths 64 (run-time length) to 1024, several instances of one length, two charge
    vectors: the batch against its instances as plans, which differ by the order of the sums."""
    import paper_0807_2387_gb300 as pkg
    rng = np.random.default_rng(5)
    dev = torch.device("cuda", 0)
    inst, q = [], []
    for k, n in enumerate((64, 32, 128, 64, 512, 32, 256)):
        s, t = (torch.tensor(rng.uniform(-0.17, 0.17, (c, 2)), device=dev) for c in (300 + 70 * k, 200 + 90 * k))
        inst.append((s, t, n, 4.0 / n))
        q.append(torch.tensor(rng.standard_normal((2, len(s))), device=dev))
    batch = pkg.FastSumBatch(inst, 2.0, 4, 2, precision=precision)
    for _ in range(2):
        phi, H = batch.eval(q, dtype=torch.float64)
    for k, (s, t, n, eps) in enumerate(inst):
        fs = pkg.FastSum(s, t, n, 2.0, 4, eps, precision=precision)
        for a, b in zip((phi[k], H[k]), fs.set_charges(q[k]).field(dtype=torch.float64)):
            assert rel(a, b) <= tol, (n, rel(a, b))
        fs.close()
    batch.close()


@pytest.mark.parametrize("n,count", [(64, 900), (256, 40000)])
def test_captured_evaluation(n, count):
    """An evaluation recorded into a graph and replayed twice with new charges: plans whose transform
    kernels are chained (n = 64) and plans without; against the same evaluations made directly."""
    import paper_0807_2387_gb300 as pkg
    rng = np.random.default_rng(6)
    dev = torch.device("cuda", 0)
    src = torch.tensor(rng.uniform(-0.17, 0.17, (count, 2)), device=dev)
    qs = torch.tensor(rng.standard_normal((3, count)), device=dev)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        fs = pkg.FastSum(src, src, n, 2.0, 4, 4.0 / n, precision=32, stream=st)
        ref = [[v.clone() for v in fs.set_charges(q).field()] for q in qs]
        q = qs[0].clone()
        phi, H = torch.empty(count, device=dev), torch.empty((count, 2), device=dev)
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            pkg.fs_set_charges(fs.handle, q)
            pkg.fs_eval_field(fs.handle, phi, H)
        for k in (2, 1):
            q.copy_(qs[k])
            graph.replay()
            st.synchronize()
            assert rel(phi, ref[k][0]) <= 2e-5 and rel(H, ref[k][1]) <= 2e-5
        for a, b in zip(fs.set_charges(qs[0]).field(), ref[0]):   # and directly again
            assert rel(a, b) <= 2e-5
    st.synchronize()
    fs.close()


@pytest.mark.parametrize("precision,tol", [(32, 2e-5), (64, 1e-12)])
@pytest.mark.parametrize("m,tile_cells", [(2, 0), (3, 4), (4, 0), (5, 0), (6, 6), (7, 0), (8, 3)])
@pytest.mark.parametrize("n_src", [1, 3, 63, 64, 65, 517])
def test_spreading_batches(n_src, m, tile_cells, precision, tol):
    """Batches of 16 or 8 sources a warp (FP32 tiles of more than 32 KB), full, partial and empty, for
    every window width: all sources in a tile or two, against direct spreading (no tiles)."""
    import paper_0807_2387_gb300 as pkg
    rng = np.random.default_rng(n_src + m)
    dev = torch.device("cuda", 0)
    src = torch.tensor(np.concatenate([rng.uniform(0.01, 0.03, (n_src, 2)), [[0.2, 0.1], [-0.2, 0.05]]]), device=dev)
    tgt = torch.tensor(rng.uniform(-0.17, 0.17, (300, 2)), device=dev)
    q = torch.tensor(rng.standard_normal(n_src + 2), device=dev)
    out = []
    for flag, tc in ((pkg.FS_FLAG_SPREAD_TILES, tile_cells), (pkg.FS_FLAG_SPREAD_DIRECT, 0)):
        fs = pkg.FastSum(src, tgt, 64, 2.0, m, 4.0 / 64, precision=precision, flags=flag, tile_cells=tc)
        out.append([v.clone() for v in fs.set_charges(q).field(dtype=torch.float64)])
        fs.close()
    for a, b in zip(*out):
        assert rel(a, b) <= tol, rel(a, b)
