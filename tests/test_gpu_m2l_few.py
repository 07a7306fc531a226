"""M2L of levels 2 .. 4 with their cells taken together, against the per-class form with the
operators as the A operand (m2l_kernel = 1): the same operands and products, so the two differ by
the order of FP32 additions only.

Cells go 384 to a set, 128 to a tile; the offsets are cut into sections by the number of sets.
Target counts lie around those sizes (every free target in a cell of its own), from one cell to
all 4,096 of level 4 and with levels below (L = 6); runs of 64 offsets' sections are the most the
form takes, 65 go per class.  Bar: sums of up to 189 x 9 p^3 products in FP32, rounded or cut at
2^-23 each in runs of a few thousand: 2e-5 of the largest component covers sqrt(n) growth with a
wide margin, an error of the index arithmetic is of order one."""
import numpy as np
import pytest

from paper_1712_07739_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ISO_C = synth.isotropic_voigt(1.0, 0.3)


def _stress(net, xt, **opt):
    import paper_1712_07739_gb300 as gb

    f = gb.FMM(precision="mixed", h_mode="iso", **opt).set_material(ISO_C)
    f.build(*(torch.tensor(a, device="cuda") for a in net))
    out = f.stress(torch.tensor(xt, device="cuda")).cpu().numpy() if xt is not None else f.nodal_forces().cpu().numpy()
    assert f.device_status() == 0
    f.close()
    return out


def _cells(net, level, n, seed):
    """n points, each in a cell of its own of the given level of the network's box."""
    x = net[0][net[1]].reshape(-1, 3)
    lo, hi = x.min(0), x.max(0)
    m, rng = 1 << level, np.random.default_rng(seed)
    c = rng.permutation(m ** 3)[:n]
    ijk = np.stack([c % m, c // m % m, c // (m * m)], 1)
    return (lo + hi) / 2 + (hi - lo).max() * 0.98 * ((ijk + 0.5) / m - 0.5)


def _close(a, b):
    assert np.abs(a - b).max() <= 2e-5 * np.abs(b).max(), np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("L", [3, 4, 5, 6])
@pytest.mark.parametrize("n", [1, 40, 64, 127, 129, 311, 384, 500, 4096])
def test_target_counts(n, L):
    net = synth.polygon_loops(n_segs=500, n_loops=20, seed=n)
    xt = _cells(net, L - 1, min(n, 8 ** (L - 1)), seed=n)
    a, b = (_stress(net, xt, p=3, levels=L, m2l_kernel=k) for k in (0, 1))
    _close(a, b)


@pytest.mark.parametrize("opt", [dict(m2l_chunks=c) for c in (0, 1, 63, 64, 65, 189)]
                         + [dict(m2l_split=s) for s in range(6)]
                         + [dict(m2l_split_levels=8), dict(m2l_split_levels=16, m2l_split_kblocks=0),
                            dict(m2l_split_levels=32), dict(m2l_basis=0), dict(m2l_svd_tol=1e-6)])
def test_options(opt):
    net = synth.polygon_loops(n_segs=900, n_loops=30, seed=5)
    a, b = (_stress(net, None, p=4, levels=6, m2l_kernel=k, **opt) for k in (0, 1))
    _close(a, b)


@pytest.mark.parametrize("p", [2, 5, 6, 7, 8])
def test_orders(p):
    net = synth.polygon_loops(n_segs=300, n_loops=10, seed=p)
    a, b = (_stress(net, None, p=p, levels=4, m2l_kernel=k) for k in (0, 1))
    _close(a, b)


@pytest.mark.parametrize("precision", ["mixed", "mixed_f64t"])
def test_repeats_bitwise(precision):
    """Sections are added in their order: two contexts give the same bits."""
    import paper_1712_07739_gb300 as gb

    net = synth.polygon_loops(n_segs=700, n_loops=20, seed=9)
    out = []
    for _ in range(2):
        f = gb.FMM(p=4, levels=5, precision=precision, h_mode="iso").set_material(ISO_C)
        f.build(*(torch.tensor(a, device="cuda") for a in net))
        out.append(f.nodal_forces().cpu().numpy())
        f.close()
    assert np.array_equal(out[0], out[1])
