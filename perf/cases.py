"""The work that programs have this library do, as cases to be timed and compared.

Each case is one call (or the one pair of calls) that a program repeats: new charges or a new magnetisation on a plan it
keeps, and the potential, the field or the gradients that come back.  Positions are the plan's, charges are the call's.

Sizes and parameters are those of this repository's workloads (``paper_0807_2387_gb300/workloads.py``) and tests.  The
radius of the near field is given in grid lines: eps_I = lines / n.  FP32 plans return float32, FP64 plans float64.
"""

import math

import numpy as np
import torch

import paper_0807_2387_gb300 as fs
from paper_0807_2387_gb300 import workloads as W

RADIUS = 0.25
#: pairs that exact() sums at most: a few seconds of float64 arithmetic
EXACT_PAIRS = 2.0e10


def listed():
    return [
        # a small problem inside somebody's larger loop: launches and latency, potential only
        dict(name="potential_1k", kind="points", n_src=1000, n_tgt=1000, same=False, mix=False, n=64, m=5, lines=4,
             precision=32, nrhs=1, q32=True, out="phi"),
        # the uniform disc of the paper's smallest test, p = 2
        dict(name="field_4k", kind="points", n_src=4096, n_tgt=4096, same=False, mix=False, n=128, m=4, lines=2,
             precision=32, nrhs=1, q32=False, out="both"),
        # an ordinary problem of odd sizes, three charge vectors on one plan, field only
        dict(name="field_100k_3rhs", kind="points", n_src=100003, n_tgt=65537, same=False, mix=False, n=512, m=5, lines=6,
             precision=32, nrhs=3, q32=True, out="H"),
        # the benchmark: 2^20 clustered sources and targets, p = 8
        dict(name="mixture_1m", kind="points", n_src=1 << 20, n_tgt=1 << 20, same=False, mix=True, n=1024, m=6, lines=8,
             precision=32, nrhs=1, q32=False, out="both"),
        # the same solve for a program whose charges and results live in page-locked host memory
        dict(name="host_300k", kind="host", n_src=300001, n_tgt=300001, same=True, mix=True, n=1024, m=6, lines=8,
             precision=32, nrhs=1, q32=True, out="both"),
        # double precision, for reference solutions and finite differences
        dict(name="field64_32k", kind="points", n_src=32768, n_tgt=32768, same=True, mix=False, n=256, m=6, lines=6,
             precision=64, nrhs=1, q32=False, out="both"),
        # one optimisation step over charges and positions: forward and every gradient
        dict(name="train_256k", kind="train", n_src=1 << 18, n_tgt=1 << 18, same=True, mix=False, n=512, m=5, lines=6,
             precision=32, nrhs=1, q32=True, out="both"),
        # one step of a micromagnetic time loop on a disc of 50,311 nodes
        dict(name="fem_disc_50k", kind="fem", rings=129, n=512, m=6, lines=6, precision=32),
        # 64 independent problems of 2^11 to 2^19 points, three charge vectors each, as one batch
        dict(name="batch_64", kind="batch", count=64, lo=11.0, hi=19.0, sizes=5, m=5, lines=6, nrhs=3, precision=32),
        # the 3D kernel on points of a ball
        dict(name="ball_256k", kind="ball", n_src=1 << 18, n_tgt=1 << 18, n=128, m=4, lines=3, precision=32),
        # one step of a 3D time loop: a cube of 384,000 tetrahedra
        dict(name="tets_384k", kind="tets", k=40, n=128, m=4, lines=3, precision=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(count):
    """The grid that the batched workload takes for `count` points, down to 64 lines."""
    return int(min(max(2 ** math.ceil(math.log2(math.sqrt(count))), 64), 1024))


def draw(rng):
    kind = rng.choice(["points", "points", "points", "points", "host", "train", "fem", "batch", "ball", "tets"])
    if kind in ("points", "host", "train"):
        precision = 64 if rng.random() < 0.2 else 32
        top = 1 << 15 if precision == 64 else 1 << 18 if kind == "train" else 1 << 20
        n_src, same = _log_int(rng, 500, top), kind == "train" or rng.random() < 0.5
        n_tgt = n_src if same else max(500, min(top, int(n_src * 2.0 ** rng.uniform(-1.5, 1.5))))
        nrhs = 3 if kind == "points" and max(n_src, n_tgt) < 200000 and rng.random() < 0.3 else 1
        return dict(kind=kind, n_src=n_src, n_tgt=n_tgt, same=same, mix=rng.random() < 0.4, n=_grid(max(n_src, n_tgt)),
                    m=rng.choice([4, 5, 6]), lines=rng.choice([4, 5, 6]), precision=precision, nrhs=nrhs,
                    q32=rng.random() < 0.5, out="both" if kind != "points" else rng.choice(["both", "both", "H", "phi"]))
    if kind == "fem":
        rings = _log_int(rng, 12, 129)
        return dict(kind=kind, rings=rings, n=min(512, 2 * _grid(3 * rings * rings)), m=rng.choice([5, 6]),
                    lines=rng.choice([4, 5, 6]), precision=32)
    if kind == "batch":
        lo = rng.uniform(9.0, 13.0)
        return dict(kind=kind, count=_log_int(rng, 3, 48), lo=lo, hi=lo + rng.uniform(1.0, 4.0), sizes=rng.randrange(1 << 20),
                    m=rng.choice([4, 5, 6]), lines=rng.choice([4, 5, 6]), nrhs=rng.choice([1, 2, 3]), precision=32)
    if kind == "ball":
        n_src = _log_int(rng, 500, 1 << 18)
        n_tgt = max(500, min(1 << 18, int(n_src * 2.0 ** rng.uniform(-1.5, 1.5))))
        return dict(kind=kind, n_src=n_src, n_tgt=n_tgt, n=128 if max(n_src, n_tgt) > 30000 else rng.choice([32, 64]), m=4,
                    lines=rng.choice([2, 3]), precision=32)
    k = _log_int(rng, 5, 40)
    return dict(kind=kind, k=k, n=128 if k > 16 else 64, m=4, lines=rng.choice([2, 3]), precision=32)


# ---------------------------------------------------------------- inputs

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _disc(g, count, mix, clusters):
    """Points in the disc: uniform, or 8 Gaussian clusters whose points outside are moved to uniform places inside."""
    def uniform(c, radius):
        u = torch.rand((2, c), generator=g, device="cuda", dtype=torch.float64)
        r, t = radius * u[0].sqrt(), 2.0 * math.pi * u[1]
        return torch.stack([r * t.cos(), r * t.sin()], 1)
    pts = uniform(count, RADIUS)
    if not mix:
        return pts
    centres, sd = clusters
    of = torch.randint(0, len(centres), (count,), generator=g, device="cuda")
    near = centres[of] + sd[of, None] * torch.randn((count, 2), generator=g, device="cuda", dtype=torch.float64)
    return torch.where((near.norm(dim=1) <= RADIUS)[:, None], near, pts).contiguous()


def _points(c, seed):
    g = _generator(seed)
    # the layouts of the sources' and the targets' clusters are not drawn: every seed asks for the same amount of work
    h = np.random.default_rng(3)
    clusters = [[torch.tensor(v, device="cuda") for v in (W.uniform_disc(h, 8, 0.15), h.uniform(0.02, 0.08, 8))] for _ in range(2)]
    src = _disc(g, c["n_src"], c["mix"], clusters[0])
    tgt = src if c["same"] else _disc(g, c["n_tgt"], c["mix"], clusters[1])
    shape = (c["n_src"],) if c["nrhs"] == 1 else (c["nrhs"], c["n_src"])
    q = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32 if c["q32"] else torch.float64)
    real = torch.float64 if c["precision"] == 64 else torch.float32
    g_phi = torch.randn((c["n_tgt"],), generator=g, device="cuda", dtype=real) if c["kind"] == "train" else None
    g_h = torch.randn((c["n_tgt"], 2), generator=g, device="cuda", dtype=real) if c["kind"] == "train" else None
    return src, tgt, q, g_phi, g_h


def _batch_sizes(c):
    rng = np.random.default_rng(c["sizes"])
    return [int(2.0 ** rng.uniform(c["lo"], c["hi"])) for _ in range(c["count"])]


def _batch(c, seed):
    g = _generator(seed)
    out = []
    for count in _batch_sizes(c):
        n = max(128, _grid(count))
        pts = _disc(g, count, False, None)
        q = torch.randn((c["nrhs"], count), generator=g, device="cuda", dtype=torch.float64)
        out.append((pts, q, n, c["lines"] / n))
    return out


def _mesh(c, seed):
    """Nodes, elements and a nodal magnetisation: uniform at some angle, with a part linear in the position."""
    rng = np.random.default_rng(seed)
    nodes, elements = W.ring_mesh(rng, c["rings"]) if c["kind"] == "fem" else W.cube_tet_mesh(rng, c["k"])
    a = rng.uniform(0.0, 2.0 * math.pi)
    mag = np.full(nodes.shape, 0.3)
    mag[:, 0], mag[:, 1] = math.cos(a) + nodes[:, 0] / 5.0, math.sin(a) + nodes[:, 1] / 5.0
    return (torch.tensor(nodes, device="cuda"), torch.tensor(elements, device="cuda"), torch.tensor(mag, device="cuda"))


def _ball(c, seed):
    g = _generator(seed)

    def ball(count):
        v = torch.randn((count, 3), generator=g, device="cuda", dtype=torch.float64)
        u = torch.rand((count, 1), generator=g, device="cuda", dtype=torch.float64)
        return (RADIUS * u ** (1.0 / 3.0) * v / v.norm(dim=1, keepdim=True)).contiguous()

    src, tgt = ball(c["n_src"]), ball(c["n_tgt"])
    return src, tgt, torch.randn((c["n_src"],), generator=g, device="cuda", dtype=torch.float64)


# ---------------------------------------------------------------- one pass

def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        inst = _batch(c, seed)
        plan = fs.FastSumBatch([(p, p, n, eps) for p, _, n, eps in inst], 2.0, c["m"], c["nrhs"], precision=c["precision"],
                               flags=fs.FS_FLAG_AUTOTUNE)
        # results side by side in two buffers, an instance's (nrhs, N) and (nrhs, N, 2) at a stretch
        counts = [c["nrhs"] * len(p) for p, _, _, _ in inst]
        phi, H = (torch.empty((sum(counts) * k,), device="cuda") for k in (1, 2))
        return dict(case=c, plan=plan, q=[q for _, q, _, _ in inst], phi=phi, H=H, phis=phi.split(counts),
                    Hs=H.split([2 * k for k in counts]))
    eps = c["lines"] / c["n"]
    if c["kind"] in ("fem", "tets"):
        nodes, elements, mag = _mesh(c, seed)
        make = fs.FastSum.fem if c["kind"] == "fem" else fs.FastSum3.fem
        return dict(case=c, plan=make(nodes, elements, c["n"], 2.0, c["m"], eps, precision=c["precision"]), mag=mag)
    if c["kind"] == "ball":
        src, tgt, q = _ball(c, seed)
        return dict(case=c, plan=fs.FastSum3(src, tgt, c["n"], 2.0, c["m"], eps, precision=c["precision"]), q=q)
    src, tgt, q, g_phi, g_h = _points(c, seed)
    state = dict(case=c, plan=fs.FastSum(src, tgt, c["n"], 2.0, c["m"], eps, precision=c["precision"]), q=q, g_phi=g_phi, g_h=g_h)
    if c["kind"] == "host":
        real = torch.float64 if c["precision"] == 64 else torch.float32
        state["q"] = q.cpu().pin_memory()
        state["phi"] = torch.empty((c["n_tgt"],), dtype=real, pin_memory=True)
        state["H"] = torch.empty((c["n_tgt"], 2), dtype=real, pin_memory=True)
    return state


def run(state):
    c, plan = state["case"], state["plan"]
    if c["kind"] == "batch":
        plan.eval_into(state["q"], state["phis"], state["Hs"])
        return {"phi": state["phi"], "H": state["H"]}
    if c["kind"] in ("fem", "tets"):
        phi, H = plan.set_magnetization(state["mag"]).field()
        return {"phi": phi, "H": H}
    if c["kind"] == "host":
        fs.fs_solve_host(plan.handle, state["q"].numpy(), state["phi"].numpy(), state["H"].numpy())
        return {"phi": state["phi"], "H": state["H"]}
    plan.set_charges(state["q"])
    if c["kind"] == "points" and c["out"] == "phi":
        return {"phi": plan.potential()}
    phi, H = plan.field(with_phi=c["kind"] != "points" or c["out"] == "both")
    if c["kind"] == "train":
        dq, dsrc, dtgt = plan.adjoint(state["g_phi"], state["g_h"], want_q=True, want_src=True, want_tgt=True)
        return {"phi": phi, "H": H, "dq": dq, "dsrc": dsrc, "dtgt": dtgt}
    return {"H": H} if phi is None else {"phi": phi, "H": H}


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Bytes: positions, charges (or magnetisation) and results once each, at the plan's precision.  Operations: the pairs
    within eps_I (a uniform density over the disc or ball; twice as many between the two sets of clusters and 3.1 times within
    one), the window's taps on both sides and the two transforms of the half of the grid that the points occupy."""
    c = case
    real = c["precision"] // 8

    def one(n_src, n_tgt, dim, n, nrhs, q_bytes, dense=1.0, backward=False, tgt_out=None, src_in=None):
        eps = c["lines"] / n
        p = max(2, c["lines"])
        pairs = float(n_src) * n_tgt * (eps / (0.25 - eps / 2)) ** dim * dense
        taps = (2 * c["m"]) ** dim
        # half of the points of the oversampled grid's active window are kept frequencies
        fft = 5.0 * n ** dim * math.log2(2 * n) * (1.5 if dim == 2 else 1.75)
        flops = pairs * (12 + 3 * p + 8 * nrhs) + nrhs * (2.0 * taps * n_src + 2.0 * (dim + 1) * taps * n_tgt + 2.0 * fft)
        moved = dim * real * (n_src + n_tgt) + (nrhs * n_src * q_bytes if src_in is None else src_in)
        moved += nrhs * n_tgt * (1 + dim) * real if tgt_out is None else tgt_out
        if backward:
            flops, moved = 3.0 * flops, moved + real * (n_tgt * (1 + 2 * dim) + n_src * (1 + dim))
        return np.array([moved, flops])

    if c["kind"] == "batch":
        got = sum(one(k, k, 2, max(128, _grid(k)), c["nrhs"], 8) for k in _batch_sizes(c))
    elif c["kind"] == "fem":
        nodes, tris = 1 + 3 * c["rings"] * (c["rings"] + 1), 6 * c["rings"] ** 2
        got = one(3 * tris + 12 * c["rings"], nodes, 2, c["n"], 1, 8, src_in=16 * nodes + 12 * tris)
    elif c["kind"] == "tets":
        nodes, tets = (c["k"] + 1) ** 3, 6 * c["k"] ** 3
        got = one(4 * tets + 36 * c["k"] ** 2, nodes, 3, c["n"], 1, 8, src_in=24 * nodes + 16 * tets)
    elif c["kind"] == "ball":
        got = one(c["n_src"], c["n_tgt"], 3, c["n"], 1, 8)
    else:
        outs = {"both": 3, "H": 2, "phi": 1}[c["out"]]
        got = one(c["n_src"], c["n_tgt"], 2, c["n"], c["nrhs"], 4 if c["q32"] else 8,
                  (3.1 if c["same"] else 2.0) if c["mix"] else 1.0, c["kind"] == "train",
                  tgt_out=c["nrhs"] * c["n_tgt"] * outs * real)
    return {"bytes": float(got[0]), "flops": float(got[1])}


# ---------------------------------------------------------------- the sums themselves, in float64

def _tiles(n_tgt, n_src):
    step = max(1, (1 << 26) // max(1, n_src))
    return [(a, min(n_tgt, a + step)) for a in range(0, n_tgt, step)]


def _sums2(x, y, q):
    """phi (R, N) and H (R, N, 2) of charges q (R, M) at y, at the targets x; a source on a target does not act on it."""
    phi, H = q.new_empty((len(q), len(x))), q.new_empty((len(q), len(x), 2))
    for a, b in _tiles(len(x), len(y)):
        d = [x[a:b, k, None] - y[None, :, k] for k in (0, 1)]
        r2 = d[0] * d[0] + d[1] * d[1]
        r2.masked_fill_(r2 == 0, math.inf)
        w = 1.0 / r2
        for k in (0, 1):
            H[:, a:b, k] = ((d[k] * w) @ q.T).T / (2.0 * math.pi)
        r2.masked_fill_(torch.isinf(r2), 1.0)
        phi[:, a:b] = (r2.log_() @ q.T).T / (-4.0 * math.pi)
    return phi, H


def _gradients2(x, y, q, g_phi, g_h):
    """dL/dq, dL/dy and dL/dx of L(phi, H) with dL/dphi = g_phi and dL/dH = g_h, for one charge vector."""
    dq, dy, dx = torch.zeros_like(q), torch.zeros_like(y), torch.zeros_like(x)
    for a, b in _tiles(len(x), 2 * len(y)):
        d = [x[a:b, k, None] - y[None, :, k] for k in (0, 1)]
        r2 = d[0] * d[0] + d[1] * d[1]
        r2.masked_fill_(r2 == 0, math.inf)
        w = 1.0 / r2
        r2.masked_fill_(torch.isinf(r2), 1.0)
        dq += g_phi[a:b] @ (r2.log_() / (-4.0 * math.pi))
        del r2
        gp, gx, gy = g_phi[a:b, None], g_h[a:b, 0, None], g_h[a:b, 1, None]
        along = (gx * d[0] + gy * d[1]) * w
        dq += along.sum(0) / (2.0 * math.pi)
        for k, gk in ((0, gx), (1, gy)):
            hess = (2.0 * along * d[k] - gk) * w          # 2 pi Hess G times g_h
            dy[:, k] += (gp * d[k] * w + hess).sum(0) * q / (2.0 * math.pi)
            dx[a:b, k] = -((gp * d[k] * w + hess) @ q) / (2.0 * math.pi)
    return dq, dy, dx


def _sums3(x, y, q):
    phi, H = q.new_empty((len(x),)), q.new_empty((len(x), 3))
    for a, b in _tiles(len(x), len(y)):
        d = [x[a:b, k, None] - y[None, :, k] for k in (0, 1, 2)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        r2.masked_fill_(r2 == 0, math.inf)
        w = r2.rsqrt_()
        phi[a:b] = (w @ q) / (4.0 * math.pi)
        w = w * w * w
        for k in (0, 1, 2):
            H[a:b, k] = ((d[k] * w) @ q) / (4.0 * math.pi)
    return phi, H


def _facets(elements):
    """The facets that one element alone has, and the node opposite each."""
    dim = elements.shape[1] - 1
    facets = torch.cat([elements[:, [j for j in range(dim + 1) if j != k]] for k in range(dim + 1)])
    opposite = torch.cat([elements[:, k] for k in range(dim + 1)])
    _, of, times = torch.unique(facets.sort(dim=1).values, dim=0, return_inverse=True, return_counts=True)
    alone = times[of] == 1
    return facets[alone], opposite[alone]


def _mesh_charges(nodes, elements, mag):
    """Quadrature points and charges of the P1 magnetisation: -div M over the elements, M . n over the boundary."""
    elements = elements.long()
    dim = nodes.shape[1]
    v, m = nodes[elements], mag[elements]
    J = v[:, 1:] - v[:, :1]                               # rows: edges from the first node
    size = torch.linalg.det(J).abs() / math.factorial(dim)
    div = torch.linalg.solve(J, m[:, 1:] - m[:, :1]).diagonal(dim1=1, dim2=2).sum(1)
    # barycentric points: one near each node of the element, and one near each node of the boundary facet
    near = 2.0 / 3.0 if dim == 2 else (5.0 + 3.0 * math.sqrt(5.0)) / 20.0
    at = nodes.new_full((dim + 1, dim + 1), (1.0 - near) / dim).fill_diagonal_(near)
    near = 0.5 + 0.5 / math.sqrt(3.0) if dim == 2 else 2.0 / 3.0
    on = nodes.new_full((dim, dim), (1.0 - near) / (dim - 1)).fill_diagonal_(near)
    facets, opposite = _facets(elements)
    f = nodes[facets]
    if dim == 2:
        e = f[:, 1] - f[:, 0]
        normal = torch.stack([e[:, 1], -e[:, 0]], 1)      # its length is the edge's
    else:
        normal = torch.linalg.cross(f[:, 1] - f[:, 0], f[:, 2] - f[:, 0]) / 2.0
    inward = ((nodes[opposite] - f[:, 0]) * normal).sum(1) > 0
    normal = torch.where(inward[:, None], -normal, normal)
    y = torch.cat([torch.einsum("pk,ekd->epd", at, v).reshape(-1, dim), torch.einsum("pk,ekd->epd", on, f).reshape(-1, dim)])
    q_in = (-div * size / (dim + 1))[:, None].expand(-1, dim + 1).reshape(-1)
    q_on = torch.einsum("pk,ekd,ed->ep", on, mag[facets], normal).reshape(-1) / dim
    return y, torch.cat([q_in, q_on])


def exact(case, seed):
    """The direct sums in float64 where they are affordable."""
    c = case
    if c["kind"] == "batch":
        if sum(float(k) * k for k in _batch_sizes(c)) > EXACT_PAIRS:
            return None
        got = [_sums2(p, p, q) for p, q, _, _ in _batch(c, seed)]
        return {"phi": torch.cat([p.reshape(-1) for p, _ in got]), "H": torch.cat([h.reshape(-1) for _, h in got])}
    if c["kind"] in ("fem", "tets"):
        elements = 6 * c["rings"] ** 2 if c["kind"] == "fem" else 6 * c["k"] ** 3
        count = 3 * c["rings"] ** 2 if c["kind"] == "fem" else (c["k"] + 1) ** 3
        if (3.0 if c["kind"] == "fem" else 4.0) * elements * count > EXACT_PAIRS:
            return None
        nodes, elements, mag = _mesh(c, seed)
        y, q = _mesh_charges(nodes, elements, mag)
        if c["kind"] == "tets":
            phi, H = _sums3(nodes, y, q)
        else:
            phi, H = (t[0] for t in _sums2(nodes, y, q[None]))
        return {"phi": phi, "H": H}
    if float(c["n_src"]) * c["n_tgt"] > EXACT_PAIRS:
        return None
    if c["kind"] == "ball":
        src, tgt, q = _ball(c, seed)
        phi, H = _sums3(tgt, src, q)
        return {"phi": phi, "H": H}
    src, tgt, q, g_phi, g_h = _points(c, seed)
    q = q.double()
    phi, H = _sums2(tgt, src, q if q.dim() == 2 else q[None])
    if q.dim() == 1:
        phi, H = phi[0], H[0]
    if c["kind"] == "train":
        dq, dsrc, dtgt = _gradients2(tgt, src, q, g_phi.double(), g_h.double())
        return {"phi": phi, "H": H, "dq": dq, "dsrc": dsrc, "dtgt": dtgt}
    if c["kind"] == "points" and c["out"] != "both":
        return {c["out"]: {"phi": phi, "H": H}[c["out"]]}
    return {"phi": phi, "H": H}
