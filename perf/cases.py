"""What is measured: the calls that a user of this package makes, over their range of sizes.

A dislocation-dynamics program keeps one context per medium and order and, at every time
step, hands it the network's current nodes, builds the tree and reads the nodal forces
(``FMM.build`` and ``FMM.nodal_forces``); less often it asks for the stress at free points
(``FMM.stress``).  An ensemble keeps a ``Batch`` and moves its nodes in place before
``Batch.step``.  The learned angular factor is evaluated (``FMM.mlp_eval``) and trained by
its gradients (``FMM.mlp_grad``).

Networks are closed polygonal glide loops with 1/2<111> Burgers vectors: "loops" with
centres uniform in the unit box and 10 to 80 segments each, "walls" with 50 segments each and
centres in Gaussian slabs (dense dislocation walls).  The plain FP64 pass returns FP64; the
mixed pass computes in FP32 with 16-bit M2L operands and its results are taken over as FP32,
as an integrator does that runs at that precision.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1712_07739_gb300 as gb
from paper_1712_07739_gb300 import synth

DEV = "cuda"
N_GAUSS = 4
MU, NU = 1.0, 0.3
ROT = synth.rotation()
VOIGT = {"iso": synth.isotropic_voigt(MU, NU), "cubic": synth.cubic_voigt(),
         "rotated": synth.rotated_voigt(synth.cubic_voigt(), ROT)}
B111 = np.array([[1, 1, 1], [-1, 1, 1], [1, -1, 1], [1, 1, -1]], dtype=np.float64) / math.sqrt(3.0)
# Chebyshev nodes with the SVD-compressed M2L, as the 1,000,000-segment workload runs it
CHEB = dict(nodes="chebyshev", m2l_svd_tol=5e-5, m2l_split=6, m2l_chunks=3, m2l_split_kblocks=1)


def _case(call, n, **kw):
    c = dict(call=call, n=n, net="loops", medium="cubic", precision="mixed", p=5, levels=4, q=32, cheb=False,
             refine=0, targets=0, networks=0)
    c.update(kw)
    return c


def listed():
    named = {
        # a single source of loops in a test cell: the smallest call, launches and host work only
        "forces_157": _case("forces", 157, p=4, levels=3, q=24),
        # the isotropic FP64 configuration of a parity study (2,000 segments, order 4)
        "forces_2k_iso_fp64": _case("forces", 2000, medium="iso", precision="fp64", p=4, levels=3),
        # a small production step in an isotropic medium
        "forces_6k_iso": _case("forces", 6011, net="walls", medium="iso", p=6, levels=5),
        # a medium-sized step in a cubic crystal with the default (dense) M2L operands
        "forces_50k": _case("forces", 50_003, p=5, levels=5),
        # dense walls, order 7 on Chebyshev nodes, uniform tree
        "forces_250k_walls": _case("forces", 250_000, net="walls", p=7, levels=6, q=16, cheb=True),
        # the largest step: a million segments, adaptive tree
        "forces_1m_walls": _case("forces", 1_000_000, net="walls", p=7, levels=7, q=16, cheb=True, refine=128),
        # the plain FP64 pass in a cubic crystal, which mixed results are checked against
        "forces_3k_fp64": _case("forces", 3_001, precision="fp64", p=5, levels=4),
        # a crystal turned off the axes: the general unit-circle rule
        "forces_6k_rotated": _case("forces", 6_101, medium="rotated", p=5, levels=4),
        # stress maps: a field sampled at free points of a network
        "stress_50k": _case("stress", 50_003, p=5, levels=5, targets=100_003),
        # an ensemble of independent networks of uneven size, stepped as one graph
        "ensemble_8": _case("ensemble", 120_001, p=6, levels=5, q=20, cheb=True, networks=8),
        # the learned angular factor: inference over many directions
        "angular_1m": _case("angular", 1_000_003),
        # the learned angular factor: one mini-batch's loss and gradient
        "angular_grad_8k": _case("angular_grad", 8192),
    }
    return [dict(c, name=k) for k, c in named.items()]


def _levels(n):
    """Depth that leaves about 4 to 34 segments per leaf of a filled box."""
    return max(3, min(7, 1 + int(round(math.log(max(n / 12.0, 64.0), 8)))))


def draw(rng):
    def log(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | 1

    kind = rng.choice(["forces", "forces", "forces", "cheb", "fp64", "general", "stress", "ensemble", "angular"])
    net = rng.choice(["loops", "walls"])
    if kind == "forces":
        n = log(150, 150_000)
        return _case("forces", n, net=net, medium=rng.choice(["iso", "cubic"]), p=rng.randint(4, 6),
                     levels=_levels(n), q=rng.choice([16, 20, 24, 32]))
    if kind == "cheb":
        n = log(20_000, 500_000)
        return _case("forces", n, net=net, p=rng.randint(5, 7), levels=_levels(n), q=rng.choice([16, 20]), cheb=True,
                     refine=rng.choice([0, 96, 128]))
    if kind == "fp64":
        n = log(150, 3_500)
        return _case("forces", n, net=net, medium=rng.choice(["iso", "cubic"]), precision="fp64",
                     p=rng.randint(4, 6), levels=_levels(n), q=rng.choice([16, 24, 32]))
    if kind == "general":
        n = log(150, 9_000)
        return _case("forces", n, net=net, medium="rotated", levels=_levels(n), q=rng.choice([20, 24, 32]))
    if kind == "stress":
        n = log(500, 50_000)
        return _case("stress", n, net=net, p=rng.randint(4, 6), levels=_levels(n), targets=log(100, 100_000),
                     medium=rng.choice(["iso", "cubic"]), q=rng.choice([16, 24, 32]))
    if kind == "ensemble":
        n = log(10_000, 110_000)
        k = rng.randint(2, 8)
        return _case("ensemble", n, p=rng.randint(5, 6), levels=_levels(n // k), q=rng.choice([16, 20]), cheb=True,
                     networks=k)
    if rng.random() < 0.5:
        return _case("angular", log(1_000, 1_000_000))
    return _case("angular_grad", log(256, 8192))


# ------------------------------------------------------------------ inputs
def _network(net, n_segs, seed):
    """Closed polygonal loops, n_segs segments in all: nodes [n, 3], segments [n, 2], Burgers vectors [n, 3]."""
    rng = np.random.default_rng(seed)
    sizes = []
    left = n_segs
    while left > 0:
        m = 50 if net == "walls" else 10 + (37 * len(sizes)) % 71
        m = left if left < m + 3 else m  # the last loop takes the remainder (at least three segments)
        sizes.append(m)
        left -= m
    sizes = np.array(sizes)
    nl = len(sizes)
    if net == "walls":
        nrm = rng.normal(size=(32, 3))
        nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
        anchor = rng.uniform(size=(32, 3))
        cen = np.zeros((0, 3))
        while len(cen) < nl:
            s = rng.integers(32, size=2 * nl)
            c = rng.uniform(size=(2 * nl, 3))
            off = np.einsum("ij,ij->i", c - anchor[s], nrm[s])
            c = c - (off - rng.normal(0.0, 0.02, 2 * nl))[:, None] * nrm[s]
            cen = np.concatenate([cen, c[np.all((c >= 0) & (c <= 1), axis=1)]])[:nl]
    else:
        cen = rng.uniform(size=(nl, 3))
    rad = np.exp(rng.uniform(math.log(0.005), math.log(0.05), nl)) * (2.0 if n_segs < 3000 else 1.0)
    bdir = B111[rng.integers(4, size=nl)] * rng.choice([-1.0, 1.0], size=nl)[:, None]
    nvec = np.cross(bdir, np.eye(3)[rng.integers(3, size=nl)])  # a {110} plane that holds b
    nvec /= np.linalg.norm(nvec, axis=1, keepdims=True)
    u = np.cross(nvec, bdir)
    loop = np.repeat(np.arange(nl), sizes)
    first = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    k = np.arange(n_segs) - first[loop]
    m = sizes[loop]
    ang = 2 * np.pi * (k + rng.uniform(-0.05, 0.05, n_segs)) / m + rng.uniform(0, 2 * np.pi, nl)[loop]
    r = rad[loop] * (1 + rng.uniform(-0.05, 0.05, n_segs))
    nodes = cen[loop] + (r * np.cos(ang))[:, None] * bdir[loop] + (r * np.sin(ang))[:, None] * u[loop]
    segs = np.stack([np.arange(n_segs), first[loop] + (k + 1) % m], 1).astype(np.int64)
    return nodes, segs, 1e-3 * bdir[loop]


def _sizes(case):
    """Segments of each network of an ensemble: uneven, in a ratio of about 1 to 8."""
    w = np.array([2.0 ** (3 * i / case["networks"]) for i in range(case["networks"])])
    return [max(500, int(case["n"] * x / w.sum())) for x in w]


def _moved(case, i, n, seed):
    """Network i of an ensemble: the same loops at every step, the nodes moved by the step's seed."""
    nodes, segs, b = _network("loops", n, 100 + i)
    return nodes + 2e-4 * np.random.default_rng([seed, i]).normal(size=nodes.shape), segs, b


def _cuda(a):
    return torch.tensor(a, device=DEV)


# A program makes its context once per medium and options and keeps it over the steps: the
# last one made is kept here, and a state holds the one that it was prepared with.
_kept = {"key": None, "handle": None}


def _handle(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "targets") and
                       (k not in ("n", "net") or case["call"] == "ensemble")))
    if _kept["key"] == key:
        return _kept["handle"]
    _kept.update(key=None, handle=None)
    kw = dict(p=case["p"], levels=case["levels"], precision=case["precision"],
              h_mode="iso" if case["medium"] == "iso" else "circle", circle_q=case["q"])
    if case["cheb"]:
        kw.update(CHEB)
    if case["call"] == "ensemble":
        h = gb.Batch(case["networks"], **kw).set_material(VOIGT[case["medium"]])
        for i, n in enumerate(_sizes(case)):
            h.build(i, *(_cuda(a) for a in _network("loops", n, 100 + i)))
    else:
        if case["refine"]:
            kw["refine_points"] = case["refine"]
        h = gb.FMM(**kw).set_material(VOIGT[case["medium"]])
    _kept.update(key=key, handle=h)
    return h


def _net_params(seed):
    """Parameters of the 3-128-128-128-27 network in the flat order of ``FMM.mlp_set``, and its output scales."""
    rng = np.random.default_rng([seed, 7])
    parts = []
    for rows, cols, fan in ((128, 3, 3), (128, 128, 128), (128, 128, 128), (32, 128, 128)):
        w = rng.normal(scale=math.sqrt(2.0 / fan), size=(rows, cols))
        b = rng.normal(scale=0.1, size=rows)
        w[27:] *= rows != 32
        b[27:] *= rows != 32
        parts += [w.ravel(), b]
    return np.concatenate(parts).astype(np.float32), rng.uniform(0.02, 0.08, 27).astype(np.float32)


def prepare(case, seed):
    if case["call"].startswith("angular"):
        h = _handle(case)
        theta, scale = _net_params(0)  # one trained network, evaluated at other directions
        h.mlp_set(theta, scale)
        g = np.random.default_rng([seed, 3])
        d = synth.directions(case["n"], seed=int(g.integers(1 << 31)))
        s = {"call": case["call"], "h": h, "dirs": _cuda(d)}
        if case["call"] == "angular_grad":
            s["y"] = _cuda(g.normal(scale=0.05, size=(case["n"], 27)).astype(np.float32))
        return s
    if case["call"] == "ensemble":
        moved = [_moved(case, i, n, seed)[0] for i, n in enumerate(_sizes(case))]
        return {"call": "ensemble", "h": _handle(case), "nodes": [_cuda(a) for a in moved]}
    s = {"call": case["call"], "h": _handle(case), "net": [_cuda(a) for a in _network(case["net"], case["n"], seed)],
         "fp64": case["precision"] == "fp64"}
    if case["call"] == "stress":
        s["x"] = _cuda(np.random.default_rng([seed, 5]).uniform(0.0, 1.0, (case["targets"], 3)))
    return s


def run(s):
    h = s["h"]
    if s["call"] == "angular":
        return h.mlp_eval(s["dirs"])
    if s["call"] == "angular_grad":
        g, loss = h.mlp_grad(s["dirs"], s["y"])
        return [g, loss]
    if s["call"] == "ensemble":
        for i, x in enumerate(s["nodes"]):
            h.nodes(i).copy_(x)
        return [f.float() for f in h.step()]
    h.build(*s["net"])
    out = h.stress(s["x"]) if s["call"] == "stress" else h.nodal_forces()
    return out if s["fp64"] else out.float()


# ------------------------------------------------------------------ the work a pass cannot do without
def _gauss():
    return np.polynomial.legendre.leggauss(N_GAUSS)


def _points(nodes, segs):
    xi, _ = _gauss()
    a, s = nodes[segs[:, 0]], nodes[segs[:, 1]] - nodes[segs[:, 0]]
    return (a[:, None, :] + (0.5 * (1 + xi))[None, :, None] * s[:, None, :]).reshape(-1, 3)


def _box_sum(g):
    """Sum over the 3 x 3 x 3 neighbourhood of every cell of a cubic grid."""
    for d in range(3):
        z = torch.zeros_like(g.narrow(d, 0, 1))
        g = g + torch.cat([g.narrow(d, 1, g.shape[d] - 1), z], d) + torch.cat([z, g.narrow(d, 0, g.shape[d] - 1)], d)
    return g


def _network_flops(case, n, seed, net):
    nodes, segs, _ = _network(net, n, seed)
    y = torch.from_numpy(_points(nodes, segs))
    lo, hi = y.amin(0), y.amax(0)
    H = float((hi - lo).amax()) * (1 + 2.0 ** -10)
    nl = 1 << (case["levels"] - 1)
    cell = ((y - (0.5 * (lo + hi) - 0.5 * H)) * (nl / H)).floor().clamp(0, nl - 1).long()
    cnt = torch.bincount((cell[:, 2] * nl + cell[:, 1]) * nl + cell[:, 0], minlength=nl ** 3).double().view(nl, nl, nl)
    if case["call"] == "stress":
        near = float(_box_sum(cnt).mean()) * case["targets"]
    else:
        near = float((cnt * _box_sum(cnt)).sum())
    pairs, occ = 0.0, (cnt > 0).double()
    while occ.shape[0] >= 4:
        m = occ.shape[0] // 2
        kids = occ.view(m, 2, m, 2, m, 2).sum((1, 3, 5))
        pairs += float((kids * _box_sum(kids)).sum() - (occ * _box_sum(occ)).sum())
        occ = (kids > 0).double()
    p = case["p"]
    # a near pair contracts 108 (isotropic 78) kernel terms; with the unit-circle rule each
    # unordered pair needs a 3 x 3 inverse per circle point; a cell pair needs the 54 products
    # per frequency of the convolution form
    pair = 202.0 if case["medium"] == "iso" else 216.0 + 15.0 * case["q"]
    return near * pair + pairs * 8 * 54 * (2 * p) ** 2 * (p + 1)


def work(case):
    n = case["n"]
    if case["call"] == "angular":
        return {"bytes": n * 30 * 4, "flops": 2.0 * n * 37_200}
    if case["call"] == "angular_grad":
        return {"bytes": n * 30 * 4 + 37_664 * 8, "flops": 6.0 * n * 37_200}
    if case["call"] == "ensemble":
        flops = sum(_network_flops(case, m, 100 + i, "loops") for i, m in enumerate(_sizes(case)))
    else:
        flops = _network_flops(case, n, 1, case["net"])
    size = 8 if case["precision"] == "fp64" else 4
    out = case["targets"] * (24 + 6 * size) if case["call"] == "stress" else n * 3 * size
    return {"bytes": n * (24 + 16 + 24) + out, "flops": flops}


# ------------------------------------------------------------------ 64-bit values, without the package's code
def _h_iso(T):
    """h_vpq = R^2 dG_vp/dx_q of the isotropic medium, the 18 components (pair, q) of the symmetric (v, p)."""
    c, a = 1.0 / (16 * math.pi * MU * (1 - NU)), 3 - 4 * NU
    for v, p in ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)):
        for q in range(3):
            s = T[v] * T[p] * (-3 * T[q])
            if v == p:
                s -= a * T[q]
            if v == q:
                s += T[p]
            if p == q:
                s += T[v]
            yield c * s


def _h_cubic(T, Q=32):
    """The same for the cubic medium with axes along x, y, z: the unit-circle integral of the Green's function."""
    C = VOIGT["cubic"]
    c12, c44 = C[0, 1], C[3, 3]
    cp, D = c12 + c44, C[0, 0] - c12 - 2 * c44
    ax = torch.stack([t.abs() for t in T]).argmin(0)
    e1 = [(ax == i).double() for i in range(3)]
    d = e1[0] * T[0] + e1[1] * T[1] + e1[2] * T[2]
    e1 = [e - d * t for e, t in zip(e1, T)]
    n = (e1[0] ** 2 + e1[1] ** 2 + e1[2] ** 2).rsqrt()
    e1 = [e * n for e in e1]
    e2 = [T[1] * e1[2] - T[2] * e1[1], T[2] * e1[0] - T[0] * e1[2], T[0] * e1[1] - T[1] * e1[0]]
    pairs = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))
    G, A, B = ([torch.zeros_like(T[0]) for _ in range(6)] for _ in range(3))
    for k in range(Q):
        c, s = math.cos(math.pi * k / Q), math.sin(math.pi * k / Q)
        z = [c * a + s * b for a, b in zip(e1, e2)]
        M = {(i, j): cp * z[i] * z[j] for i, j in pairs}
        for i in range(3):
            M[i, i] = M[i, i] + (c44 + D * z[i] * z[i])
        adj = {(0, 0): M[1, 1] * M[2, 2] - M[1, 2] ** 2, (1, 1): M[0, 0] * M[2, 2] - M[0, 2] ** 2,
               (2, 2): M[0, 0] * M[1, 1] - M[0, 1] ** 2, (1, 2): M[0, 1] * M[0, 2] - M[0, 0] * M[1, 2],
               (0, 2): M[0, 1] * M[1, 2] - M[0, 2] * M[1, 1], (0, 1): M[0, 2] * M[1, 2] - M[0, 1] * M[2, 2]}
        w = (M[0, 0] * adj[0, 0] + M[0, 1] * adj[0, 1] + M[0, 2] * adj[0, 2]).reciprocal()
        inv = [[adj[min(i, j), max(i, j)] * w for j in range(3)] for i in range(3)]
        # F = inv [(zT) + (Tz)] inv, with (zT) + (Tz) = cp (z T' + T z') + 2 D diag(z T)
        iz = [sum(inv[i][j] * z[j] for j in range(3)) for i in range(3)]
        it = [sum(inv[i][j] * T[j] for j in range(3)) for i in range(3)]
        e = [2 * D * z[j] * T[j] for j in range(3)]
        for m, (i, j) in enumerate(pairs):
            f = cp * (iz[i] * it[j] + it[i] * iz[j]) + sum(inv[i][l] * e[l] * inv[l][j] for l in range(3))
            G[m] += inv[i][j]
            A[m] += c * f
            B[m] += s * f
    for m in range(6):
        for q in range(3):
            yield (e1[q] * A[m] + e2[q] * B[m] - T[q] * G[m]) / (4 * math.pi * Q)


def _levi(i, j, k):
    return (i - j) * (j - k) * (k - i) / 2


def _direct_stress(medium, x, own, y, q, seg):
    """sum_j K(x_i - y_j) q_j over all source points not on the target's own segment (own < 0: none is left out)."""
    vi = {(0, 0): 0, (1, 1): 1, (2, 2): 2, (1, 2): 3, (2, 1): 3, (0, 2): 4, (2, 0): 4, (0, 1): 5, (1, 0): 5}
    pairs = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))
    Cv = VOIGT[medium]
    C = np.array([[[[Cv[vi[i, j], vi[k, l]] for l in range(3)] for k in range(3)] for j in range(3)] for i in range(3)])
    eps = np.array([[[_levi(i, j, k) for k in range(3)] for j in range(3)] for i in range(3)])
    A = np.einsum("ngr,abvg,pqwn->abwrvpq", eps, C, C)
    As = np.zeros((6, 9, 18))
    for a, (i, j) in enumerate(pairs):
        for m, (v, p) in enumerate(pairs):
            t = A[i, j, :, :, v, p, :] + (A[i, j, :, :, p, v, :] if v != p else 0.0)
            As[a, :, 3 * m:3 * m + 3] = t.reshape(9, 3)
    P = torch.einsum("jw,awk->kja", q, _cuda(As)).contiguous()  # [18, N, 6]
    out = torch.zeros(len(x), 6, dtype=torch.float64, device=DEV)
    step = max(1, int(6e6) // len(y))
    for i0 in range(0, len(x), step):
        xs = x[i0:i0 + step]
        d = [xs[:, None, i] - y[None, :, i] for i in range(3)]
        r2 = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
        r2[own[i0:i0 + step, None] == seg[None, :]] = math.inf
        w = r2.reciprocal()
        ir = torch.where(torch.isinf(r2), torch.ones_like(r2), r2).rsqrt()
        T = [v * ir for v in d]
        for k, h in enumerate(_h_iso(T) if medium == "iso" else _h_cubic(T)):
            out[i0:i0 + step] += (h * w) @ P[k]
    return out


def _exact_network(case, nodes, segs, b, x):
    # in the rotated crystal: the cubic medium's problem in the crystal's own axes
    rot = ROT if case["medium"] == "rotated" else np.eye(3)
    medium = "cubic" if case["medium"] == "rotated" else case["medium"]
    nodes, b = nodes @ rot, b @ rot
    _, wq = _gauss()
    s = nodes[segs[:, 1]] - nodes[segs[:, 0]]
    q = 0.5 * wq[None, :, None, None] * b[:, None, :, None] * s[:, None, None, :]
    y, q = _cuda(_points(nodes, segs)), _cuda(q.reshape(-1, 9))
    seg = torch.arange(len(segs), device=DEV).repeat_interleave(N_GAUSS)
    if x is not None:
        return _direct_stress(medium, _cuda(x @ rot), torch.full((len(x),), -1, device=DEV), y, q, seg)
    sig = _direct_stress(medium, y, seg, y, q, seg).view(-1, N_GAUSS, 6)
    bb, ss, xi, wt = _cuda(b), _cuda(s), _cuda(_gauss()[0]), _cuda(wq)
    full = sig[..., [0, 5, 4, 5, 1, 3, 4, 3, 2]].view(-1, N_GAUSS, 3, 3)
    pk = torch.linalg.cross(torch.einsum("sgij,sj->sgi", full, bb), ss[:, None, :].expand(-1, N_GAUSS, 3), dim=-1)
    f = torch.zeros(len(nodes), 3, dtype=torch.float64, device=DEV)
    for col, shape in ((0, 1 - xi), (1, 1 + xi)):
        f.index_add_(0, _cuda(segs[:, col]), torch.einsum("g,sgi->si", 0.25 * wt * shape, pk))
    return f @ _cuda(rot.T.copy())


def _exact_angular(case, seed):
    theta, scale = _net_params(0)
    g = np.random.default_rng([seed, 3])
    d = _cuda(synth.directions(case["n"], seed=int(g.integers(1 << 31)))).double()
    w, o = [], 0
    for rows, cols in ((128, 3), (128, 128), (128, 128), (32, 128)):  # weights are BF16 numbers, biases FP32
        W = _cuda(theta[o:o + rows * cols]).bfloat16().double().view(rows, cols).requires_grad_(True)
        o += rows * cols
        b = _cuda(theta[o:o + rows]).double().requires_grad_(True)
        o += rows
        w.append((W, b))
    up = (d[:, 2] > 0) | ((d[:, 2] == 0) & ((d[:, 1] > 0) | ((d[:, 1] == 0) & (d[:, 0] >= 0))))
    sign = torch.where(up, 1.0, -1.0).double()[:, None]
    a = sign * d
    for W, b in w[:3]:
        a = torch.nn.functional.silu(a @ W.T + b)
    out = (a @ w[3][0].T + w[3][1])[:, :27]
    sc = _cuda(scale).double()
    if case["call"] == "angular":
        return (sign * sc * out).detach()
    y = _cuda(g.normal(scale=0.05, size=(case["n"], 27)).astype(np.float32)).double()
    loss = ((out - sign * y / sc) ** 2).mean()
    loss.backward()
    return [torch.cat([t.grad.reshape(-1) for pair in w for t in pair]), float(loss.detach())]


def exact(case, seed):
    """The direct sum over all pairs where that takes seconds; the network by plain FP64 arithmetic."""
    if case["call"].startswith("angular"):
        return _exact_angular(case, seed)
    most = 150_000 if case["medium"] == "iso" else 24_500
    if case["call"] == "stress":
        x = np.random.default_rng([seed, 5]).uniform(0.0, 1.0, (case["targets"], 3))
        pairs = len(x) * case["n"] * N_GAUSS
        return _exact_network(case, *_network(case["net"], case["n"], seed), x) if pairs <= most ** 2 else None
    if case["call"] == "ensemble":
        if sum(n * n for n in _sizes(case)) * N_GAUSS ** 2 > most ** 2:
            return None
        return [_exact_network(case, *_moved(case, i, n, seed), None) for i, n in enumerate(_sizes(case))]
    if case["n"] * N_GAUSS > most:
        return None
    return _exact_network(case, *_network(case["net"], case["n"], seed), None)
