"""The near field with the learned factor."""
import numpy as np
import pytest

from paper_1712_07739_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MEDIA = {"cubic": synth.cubic_voigt(), "soft": synth.cubic_voigt(2.37, 1.11, 0.3),
         "turned": synth.rotated_voigt(synth.cubic_voigt(), synth.rotation())}


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
