"""Network evaluation and gradient at the sizes where their tiles can go wrong: 16 directions a
warp, 8 or 2 warps a block, blocks striding over the tiles, gradient runs of 128 samples up to 64
runs, then longer ones.

Evaluation: a direction's outputs do not depend on its place in the call, so any n gives the bits
of the same rows in another call; against the FP64 reference with BF16 weights the activations'
rounding (2^-9 each, three layers, the largest of many components) stays below 5e-2 of the largest
output, an index error is of order one.  Gradient: per layer within 1e-1 of the reference's norm
(a few per cent from BF16 activations and gradients at a handful of samples), repeated bitwise."""
import numpy as np
import pytest

from oracle import mlp_ref
from paper_1712_07739_gb300 import synth
from test_gpu_mlp import _ctx, _params, _rounded

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 8, 9, 15, 16, 17, 127, 128, 129, 2048, 38_911, 38_913, 80_000])
def test_eval_sizes(n):
    f = _ctx()
    theta, scale = _params(n)
    f.mlp_set(theta, scale)
    d = synth.directions(n, seed=n)
    dirs = torch.tensor(d, device="cuda")
    h = f.mlp_eval(dirs)
    k = min(n, 1500)
    pick = np.unique(np.concatenate([np.arange(n - k // 2, n), np.random.default_rng(n).integers(0, n, k)]))
    again = f.mlp_eval(dirs[torch.tensor(pick, device="cuda")].contiguous()).cpu().numpy()
    h = h.cpu().numpy()
    assert np.array_equal(h[pick], again)
    ref, _ = mlp_ref.forward(_rounded(theta), d[pick].astype(np.float64), scale)
    assert np.abs(again - ref).max() <= 5e-2 * np.abs(ref).max()


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 33, 127, 128, 129, 1000, 8191, 8192, 8193, 20_000])
def test_gradient_sizes(n):
    f = _ctx()
    theta, scale = _params(n)
    f.mlp_set(theta, scale)
    dirs = synth.directions(n, seed=n)
    y = np.random.default_rng(n).normal(scale=0.05, size=(n, 27)).astype(np.float32)
    args = torch.tensor(dirs, device="cuda"), torch.tensor(y, device="cuda")
    g, loss = f.mlp_grad(*args)
    g2, loss2 = f.mlp_grad(*args)
    assert loss == loss2 and torch.equal(g, g2)
    g = g.cpu().numpy().astype(np.float64)
    l_ref, g_ref = mlp_ref.loss_and_grad(_rounded(theta), dirs.astype(np.float64), y.astype(np.float64), scale)
    assert abs(loss - l_ref) <= 5e-2 * l_ref
    o = 0
    for name, shp in mlp_ref.SIZES:
        m = int(np.prod(shp))
        a, b = g[o:o + m], g_ref[o:o + m]
        assert np.linalg.norm(a - b) <= 1e-1 * np.linalg.norm(b), name
        o += m
