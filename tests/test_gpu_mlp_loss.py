"""The loss of a batch against the same sum in FP64 over the outputs of the network evaluation.

Both run the same four layers, so only the loss's own arithmetic differs.  Its terms take about five
FP32 roundings (the reference's outputs one for their scale), of either sign and independent: 1e-7
of a term, below 5e-7 / sqrt(n) of the mean with a wide margin; the returned number is rounded to
FP32 (6e-8).  Bar 1e-7 + 5e-7 / sqrt(n); summed in FP32 one sample after the other, 8,192 samples
are up to 2e-6 off."""
import numpy as np
import pytest

from paper_1712_07739_gb300 import synth
from test_gpu_mlp import _ctx, _params

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 17, 512, 4097, 8192, 300_000])
def test_loss_is_the_fp64_sum(n, seed):
    f = _ctx()
    theta, scale = _params(seed)
    f.mlp_set(theta, scale)
    dirs = torch.tensor(synth.directions(n, seed=seed + 50), device="cuda")
    y = torch.tensor(np.random.default_rng(seed).normal(scale=0.05, size=(n, 27)).astype(np.float32), device="cuda")
    _, loss = f.mlp_grad(dirs, y)
    want = float((((f.mlp_eval(dirs).double() - y.double()) / torch.tensor(scale, device="cuda").double()) ** 2).mean())
    assert abs(loss - want) <= (1e-7 + 5e-7 / n ** 0.5) * want, loss / want - 1
