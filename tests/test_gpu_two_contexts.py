"""Two contexts of one process with different M2L operand modes: which residual operator an offset
has belongs to the context, so each gives the bits it gives alone, whichever was set up last."""
import numpy as np
import pytest

from paper_1712_07739_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _make(split, kernel, net):
    import paper_1712_07739_gb300 as gb

    f = gb.FMM(p=4, levels=6, precision="mixed", h_mode="iso", m2l_split=split, m2l_kernel=kernel).set_material(
        synth.isotropic_voigt(1.0, 0.3))
    f.build(*(torch.tensor(a, device="cuda") for a in net))
    return f


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("pair", [(6, 4), (4, 6), (0, 2), (5, 6), (6, 5)])
def test_split_modes_side_by_side(pair, kernel):
    net = synth.polygon_loops(n_segs=900, n_loops=30, seed=5)
    x = torch.tensor(np.random.default_rng(1).uniform(0.1, 0.9, (2000, 3)), device="cuda")
    alone = []
    for s in pair:
        f = _make(s, kernel, net)
        alone.append(f.stress(x).cpu().numpy())
        f.close()
    both = [_make(s, kernel, net) for s in pair]
    for f, want in zip(both, alone):
        assert np.array_equal(f.stress(x).cpu().numpy(), want)
        assert f.device_status() == 0
    assert not np.array_equal(*alone)
