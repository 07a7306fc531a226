"""Near field at the sizes where its work plan and tiles can go wrong, against the oracle's
Lagrange FMM on the same tree.

Target blocks hold 64 points and list tiles 32 entries, chunks are powers of two, items are cut
at a few hundred pairs when the network is small, and the circle rule pairs the points phi and
-phi: segment counts from one up, point counts around 32 and 64 in one leaf, and rules of 1, 2,
odd, even and more points than the shared table holds.  The FP64 pass runs the same plan in FP64,
so its bar is the FP64 path's 1e-10 (rounding only; an index error is of order one); the mixed
pass adds FP32 rounding and the M2L's 16-bit operands, bar 1e-4.  Free targets lie outside the
root cube too, where the local expansions extrapolate: FP64 only."""
import numpy as np
import pytest

import oracle
from oracle import oracle_b
from paper_1712_07739_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MEDIA = {"iso": (synth.isotropic_voigt(1.0, 0.3), "iso"), "cubic": (synth.cubic_voigt(), "circle"),
         "soft": (synth.cubic_voigt(2.37, 1.11, 0.3), "circle"),  # Zener ratio 0.48
         "turned": (synth.rotated_voigt(synth.cubic_voigt(), synth.rotation()), "circle")}


def _network(sizes, seed, spread):
    """Loops of the given sizes near a few places: crowded leaves beside empty ones."""
    rng = np.random.default_rng(seed)
    nodes, segs, b, base = [], [], [], 0
    for k, m in enumerate(sizes):
        c = np.array([0.2, 0.7, 0.45])[(k + np.arange(3)) % 3] + spread * rng.normal(size=3)
        ang = 2 * np.pi * (np.arange(m) + 0.2 * rng.random(m)) / max(m, 2)
        u = np.linalg.qr(rng.normal(size=(3, 3)))[0]
        r = 0.03 + 0.05 * rng.random()
        nodes.append(c + r * (np.cos(ang)[:, None] * u[0] + np.sin(ang)[:, None] * u[1]))
        if m == 1:  # a single open segment
            nodes[-1] = np.stack([c, c + 0.1 * u[0]])
            segs.append([[base, base + 1]])
        else:
            segs.append([[base + i, base + (i + 1) % m] for i in range(m)])
        b.append(np.repeat((1e-3 * u[2])[None], m, 0))
        base += len(nodes[-1])
    return np.concatenate(nodes), np.concatenate(segs).astype(np.int64), np.concatenate(b)


def _run(net, medium, Q, precision, xt=None, p=3, L=3):
    import paper_1712_07739_gb300 as gb

    nodes, segs, b = net
    C, mode = MEDIA[medium]
    f = gb.FMM(p=p, levels=L, precision=precision, h_mode=mode, circle_q=Q).set_material(C)
    f.build(*(torch.tensor(a, device="cuda") for a in net))
    mat = oracle.Material.iso(1.0, 0.3) if mode == "iso" else oracle.Material.aniso(C, Q=Q)
    y, q, sid = oracle.quadrature(nodes, segs, b, 4)
    if xt is None:
        got = f.nodal_forces().cpu().numpy()
        want = oracle.nodal_forces(nodes, segs, b, oracle_b.lagrange_fmm(mat, y, q, sid, p=p, L=L), 4)
    else:
        got = f.stress(torch.tensor(xt, device="cuda")).cpu().numpy()
        want = oracle_b.lagrange_fmm(mat, y, q, sid, p=p, L=L, xt=xt, tseg=-np.ones(len(xt), np.int64))
    assert f.device_status() == 0
    f.close()
    return oracle.rel_l2(got, want)


@pytest.mark.parametrize("precision,bar", [("fp64", 1e-10), ("mixed", 1e-4)])
@pytest.mark.parametrize("medium", list(MEDIA))
@pytest.mark.parametrize("sizes", [(1, 1), (3,), (8, 1), (9, 7), (15, 16, 17), (64, 33, 5), (90, 80, 70)])
def test_leaf_populations(sizes, medium, precision, bar):
    err = _run(_network(sizes, seed=sum(sizes), spread=0.02), medium, 12, precision)
    assert err <= bar, err


@pytest.mark.parametrize("medium", ["cubic", "turned"])
@pytest.mark.parametrize("Q", [1, 2, 3, 4, 5, 16, 17, 64, 601, 1030])
def test_circle_points(Q, medium):
    """Both precisions: the FP64 pass in moment form, the mixed pass (pointwise in the turned
    crystal); 601 and 1,030 points are beyond the shared tables."""
    net = _network((6, 5, 4), seed=Q, spread=0.05)
    assert _run(net, medium, Q, "fp64") <= 1e-10
    assert _run(net, medium, Q, "mixed") <= 1e-4


@pytest.mark.parametrize("medium", ["iso", "cubic", "turned"])
@pytest.mark.parametrize("n_t", [1, 31, 64, 65, 200])
def test_free_targets(n_t, medium):
    net = _network((40, 33, 21), seed=n_t, spread=0.05)
    rng = np.random.default_rng(n_t)
    xt = 0.45 + 0.35 * rng.normal(size=(n_t, 3))
    assert _run(net, medium, 16, "fp64", xt) <= 1e-10
