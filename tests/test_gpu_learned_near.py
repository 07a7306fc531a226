"""The learned near field against a restatement on the CPU.

What the pair kernel uses of the network is one quadratic per angular bin and component, fitted to
the network's values at 8 x 8 directions.  The restatement fits the same quadratics in FP64 to
mlp_eval's values and sums, over the near pairs that take the network, the difference between
learned and plain kernel; on the GPU that is the stress with some bins accepted less the stress with
every bin on the plain rule, in which the far field and all other pairs cancel.  Bar per point:
5e-6 of the sum of the magnitudes of all products of its pairs.  That covers FP32 values whose
place in the bin carries 2e-6 of its width (a direction's FP32 rounding, 1.2e-7, beside a bin of
1/8 to 1/16) and whose coefficients and contraction carry 1e-6; one lost, doubled or misplaced pair
of a few hundred is of order 1e-3."""
import numpy as np
import pytest

import oracle
from paper_1712_07739_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MEDIA = {"cubic": synth.cubic_voigt(), "soft": synth.cubic_voigt(2.37, 1.11, 0.3),
         "turned": synth.rotated_voigt(synth.cubic_voigt(), synth.rotation())}
PAIRS = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))
PER = 8
GRID = (2.0 * np.arange(PER) + 1.0) / PER - 1.0
M2 = float((GRID ** 2).mean())


def _fold(d):
    up = (d[:, 2] > 0) | ((d[:, 2] == 0) & ((d[:, 1] > 0) | ((d[:, 1] == 0) & (d[:, 0] >= 0))))
    return np.where(up, 1.0, -1.0)


def _bins(d):
    """Bin (face of the dominant axis, 16 x 16), place in it and sign of the fold."""
    sg = _fold(d)
    x, y, z = (sg[:, None] * d).T
    a = np.abs([x, y, z])
    top = (a[2] >= a[0]) & (a[2] >= a[1])
    side = ~top & (a[0] >= a[1])
    f = np.where(top, 0, np.where(side, np.where(x > 0, 1, 2), np.where(y > 0, 3, 4)))
    p = np.where(side, y, x)
    q = np.where(top, y, z)
    m = np.where(top, a[2], np.where(side, a[0], a[1]))
    tp, tq = (p / m + 1.0) * 8.0, (q / m + 1.0) * 8.0
    bu, bv = np.clip(tp.astype(int), 0, 15), np.clip(tq.astype(int), 0, 15)
    return f * 256 + bu * 16 + bv, 2.0 * (tp - bu) - 1.0, 2.0 * (tq - bv) - 1.0, sg


def _directions(u, v):
    """Unit directions at the places (u, v) of every bin, [1280, len(u), 3]."""
    b = np.arange(1280)
    p = -1.0 + (2.0 * ((b // 16) % 16)[:, None] + 1.0 + u[None, :]) / 16.0
    q = -1.0 + (2.0 * (b % 16)[:, None] + 1.0 + v[None, :]) / 16.0
    f, one = (b // 256)[:, None], np.ones_like(p)
    d = np.stack([np.where((f == 0) | (f >= 3), p, np.where(f == 1, one, -one)),
                  np.where(f == 0, q, np.where(f <= 2, p, np.where(f == 3, one, -one))),
                  np.where(f == 0, one, q)], -1)
    return d / np.linalg.norm(d, axis=-1, keepdims=True)


def _basis(u, v):
    return np.stack([np.ones_like(u), u, v, u * u - M2, u * v, v * v - M2], -1)


U8, V8 = np.tile(GRID, PER), np.repeat(GRID, PER)


def _ev(fn, d):
    flat = d.reshape(-1, 3).astype(np.float32)
    return fn(torch.tensor(flat, device="cuda")).cpu().numpy().astype(np.float64).reshape(d.shape[:-1] + (27,))


def _symmetric(h27):
    h = h27.reshape(h27.shape[:-1] + (3, 3, 3))
    return np.stack([0.5 * (h[..., v, p, q] + h[..., p, v, q]) for v, p in PAIRS for q in range(3)], -1)


def _tables(f):
    """Coefficients [1280, 6, 18] and, per bin, the largest errors of the network and of the polynomial."""
    grid = _directions(U8, V8)
    net, plain = _ev(f.mlp_eval, grid), _ev(f.mlp_labels, grid)
    B = _basis(U8, V8)
    coef = np.einsum("gc,bgk->bck", B, _symmetric(net)) / (B * B).sum(0)[None, :, None]
    rms = np.sqrt((plain ** 2).mean())
    e_net = np.abs(net - plain).max((1, 2)) / rms
    w = np.linspace(-1.0, 1.0, 5)
    u, v = np.concatenate([U8, np.tile(w, 5)]), np.concatenate([V8, np.repeat(w, 5)])
    far = _symmetric(_ev(f.mlp_labels, _directions(u, v)))
    e_poly = np.abs(np.einsum("gc,bck->bgk", _basis(u, v), coef) - far).max((1, 2)) / rms
    return coef, e_net, e_poly


def _contraction(C):
    """K_abwr = sum_k A[ab, wr, k] h_k / R^2 over the 18 components of the symmetric h."""
    Cf = oracle.voigt_to_cijkl(C)
    eps = np.array([[[(i - j) * (j - k) * (k - i) / 2 for k in range(3)] for j in range(3)] for i in range(3)])
    A = np.einsum("ngr,abvg,pqwn->abwrvpq", eps, Cf, Cf)
    out = np.zeros((6, 9, 18))
    for a, (i, j) in enumerate(PAIRS):
        for m, (v, p) in enumerate(PAIRS):
            t = A[i, j, :, :, v, p, :] + (A[i, j, :, :, p, v, :] if v != p else 0.0)
            out[a, :, 3 * m:3 * m + 3] = t.reshape(9, 3)
    return out


def _segments(m, seed, close=False):
    """Short open segments (one Gauss point each) in three neighbouring leaves of the unit box, m in the
    first; two at its corners.  close: the first two of them 2e-6 apart."""
    rng = np.random.default_rng(seed)
    mid = [[[0.0, 0.0, 0.0]], [[1.0, 1.0, 1.0]]]
    for c, k in (((0.38, 0.4, 0.38), m), ((0.62, 0.4, 0.38), 33), ((0.62, 0.62, 0.62), 20)):
        mid.append(np.array(c) + rng.uniform(-0.1, 0.1, (k, 3)))
    mid = np.concatenate([np.array(x) for x in mid])
    if close:
        mid[3] = mid[2] + [0.0, 0.0, 2e-6]
    t = rng.normal(size=mid.shape)
    t *= 0.004 / np.linalg.norm(t, axis=1, keepdims=True)
    t[:2] *= 1e-3
    nodes = np.stack([mid - t / 2, mid + t / 2], 1).reshape(-1, 3)
    n = len(mid)
    return nodes, np.arange(2 * n).reshape(n, 2).astype(np.int64), 1e-3 * rng.normal(size=(n, 3))


def _context(C, net=None, seed=0, **kw):
    import paper_1712_07739_gb300 as gb

    f = gb.FMM(p=3, levels=3, n_gauss=1, precision="mixed", h_mode="mlp", circle_q=24, mlp_min_dist=3.0,
               **kw).set_material(C)
    rng = np.random.default_rng(seed)
    f.mlp_set(rng.normal(scale=0.1, size=gb.MLP_PARAMS).astype(np.float32),
              rng.uniform(0.05, 0.1, 27).astype(np.float32))
    if net is not None:
        f.build(*(torch.tensor(a, device="cuda") for a in net))
    return f


def _stress(f, n, x):
    if x is not None:
        return f.stress(torch.tensor(x, device="cuda")).cpu().numpy()
    s = torch.empty((n, 6), dtype=torch.float64, device="cuda")
    f.nodal_forces(sigma_pts=s)
    return s.cpu().numpy()


def _restated(f, C, net, x, accepted, coef):
    """Sum over the pairs that take the network of learned less plain stress, and of the magnitudes."""
    nodes, segs, b = net
    S = nodes[segs[:, 1]] - nodes[segs[:, 0]]
    y = nodes[segs[:, 0]] + 0.5 * S
    own = np.arange(len(y)) if x is None else np.full(len(x), -1)
    tl = np.linalg.norm(S, axis=1) if x is None else np.zeros(len(x))
    xt = y if x is None else x
    H = (y.max(0) - y.min(0)).max() * (1 + 2.0 ** -10)
    o = 0.5 * (y.max(0) + y.min(0)) - 0.5 * H

    def leaf(z):
        return np.clip(np.floor((z - o) * (4 / H)).astype(int), 0, 3)

    i, j = np.nonzero((np.abs(leaf(xt)[:, None] - leaf(y)[None]).max(-1) <= 1) & (own[:, None] != np.arange(len(y))))
    d = xt[i] - y[j]
    r = np.linalg.norm(d, axis=1)
    keep = r >= 3.0 * np.maximum(tl[i], np.linalg.norm(S, axis=1)[j])
    i, j, d, r = i[keep], j[keep], d[keep], r[keep]
    bin_, u, v, sg = _bins(d)
    keep = accepted[bin_]
    i, j, d, r, bin_, u, v, sg = (a[keep] for a in (i, j, d, r, bin_, u, v, sg))
    learned = sg[:, None] * np.einsum("nc,nck->nk", _basis(u, v), coef[bin_])
    plain = _symmetric(_ev(f.mlp_labels, d / r[:, None]))
    q = np.einsum("nw,nr->nwr", b, S).reshape(-1, 9)  # one Gauss point: half its weight 2
    A = _contraction(C)
    diff = np.einsum("awk,nk,nw->na", A, learned - plain, q[j]) / (r * r)[:, None]
    size = np.einsum("awk,nk,nw->na", np.abs(A), np.abs(learned) + np.abs(plain), np.abs(q[j])) / (r * r)[:, None]
    out, mag = np.zeros((len(xt), 6)), np.zeros((len(xt), 6))
    np.add.at(out, i, diff)
    np.add.at(mag, i, size)
    return out, mag.max(1, keepdims=True), len(i)


@pytest.mark.parametrize("part", [1.0, 0.5])  # share of the bins that the network serves (about)
@pytest.mark.parametrize("free", [False, True])
@pytest.mark.parametrize("medium", ["cubic", "turned"])
@pytest.mark.parametrize("m", [1, 31, 32, 33, 63, 64, 65, 200])
def test_learned_pairs(m, medium, free, part):
    C, net = MEDIA[medium], _segments(m, seed=m)
    x = np.array([0.42, 0.45, 0.42]) + np.random.default_rng(m + 1).uniform(-0.15, 0.15, (m, 3)) if free else None
    f = _context(C, net, seed=m)
    coef, e_net, e_poly = _tables(f)
    err = np.sort(np.maximum(e_net, e_poly))
    # the widest gap near the middle: no bin whose side FP32 could change
    k = 513 + int(np.argmax(np.diff(err[512:769])))
    tol = 1e30 if part == 1.0 else 0.5 * (err[k - 1] + err[k])
    f.mlp_calibrate(tol)
    got = _stress(f, len(net[1]), x)
    f.mlp_calibrate(1e-30)
    got = got - _stress(f, len(net[1]), x)
    want, mag, n = _restated(f, C, net, x, np.maximum(e_net, e_poly) <= tol, coef)
    f.close()
    assert n > 3 * m
    assert np.all(np.abs(got - want) <= 5e-6 * mag + 1e-300), np.max(np.abs(got - want) / np.maximum(mag, 1e-300))


def test_learned_sum_beside_a_close_pair():
    """A pair 2e-6 apart adds a stress 1e4 and more times the learned pairs' to its two points; what these
    add must not be rounded to the digits of that."""
    C, net = MEDIA["cubic"], _segments(64, seed=5, close=True)
    f = _context(C, net, seed=5)
    coef, _, _ = _tables(f)
    f.mlp_calibrate(1e30)
    got = _stress(f, len(net[1]), None)
    f.mlp_calibrate(1e-30)
    plain = _stress(f, len(net[1]), None)
    want, mag, _ = _restated(f, C, net, None, np.ones(1280, bool), coef)
    f.close()
    assert np.abs(plain[2:4]).max() > 1e4 * mag[2:4].max()
    assert np.all(np.abs(got - plain - want) <= 5e-6 * mag + 1e-11 * np.abs(plain).max(1, keepdims=True))


def test_calibration_judges_the_polynomials():
    """A bin is flagged by the larger of two errors, the network's at 64 directions and its
    polynomial's at these and at 25 more from edge to edge, both against the plain rule.  In a
    crystal of Zener ratio 8 the two judge many bins differently at some tolerance."""
    import paper_1712_07739_gb300 as gb

    f = gb.FMM(p=3, levels=3, precision="mixed", h_mode="mlp", circle_q=32).set_material(
        synth.cubic_voigt(1.684, 1.214, 1.88))
    f.mlp_train(torch.tensor(synth.directions(300_000, seed=1), device="cuda"), epochs=15, batch=4096, lr=3e-3, seed=4)
    _, e_net, e_poly = _tables(f)
    both = np.maximum(e_net, e_poly)
    tols = np.geomspace(np.quantile(both, 0.02), both.max(), 400)
    gap = [(both > t).sum() - (e_net > t).sum() for t in tols]
    tol = tols[int(np.argmax(gap))]
    print(f"bins flagged at {tol:.3e}: by the network {(e_net > tol).sum()}, by either {(both > tol).sum()}")
    assert max(gap) >= 8
    near = np.sum(np.abs(both / tol - 1.0) < 1e-4)  # bins that FP32 could put on the other side
    assert abs(f.mlp_calibrate(tol) * 1280 - (both > tol).sum()) <= near


def test_force_call_after_new_network_under_capture():
    """Setting a network leaves nothing for the force call to prepare: it neither allocates nor
    synchronises, so it can be captured, and it uses the new network."""
    import paper_1712_07739_gb300 as gb

    rng = np.random.default_rng(9)
    second = rng.normal(scale=0.1, size=gb.MLP_PARAMS).astype(np.float32), rng.uniform(0.05, 0.1, 27).astype(np.float32)
    net = _segments(40, seed=1)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        f = _context(MEDIA["cubic"], net, stream=s)
        f.mlp_calibrate(1e30)
        out = f.nodal_forces()
        f.mlp_set(*second)
    s.synchronize()
    first, out = out.cpu().numpy(), torch.zeros_like(out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        f.nodal_forces(out=out)
    graph.replay()
    torch.cuda.synchronize()
    again = f.nodal_forces()
    torch.cuda.synchronize()
    again, out = again.cpu().numpy(), out.cpu().numpy()
    assert np.abs(out - again).max() <= 1e-12 * np.abs(again).max()
    assert np.abs(first - again).max() > 1e-3 * np.abs(again).max()
