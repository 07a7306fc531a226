"""The field of a built network is the field at its build: a caller that moves its nodes on, or
reuses its arrays, before the next build still gets it at free points."""
import numpy as np
import pytest

from paper_1712_07739_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,mode", [("fp64", "iso"), ("fp64", "circle"), ("mixed", "iso"), ("mixed", "circle")])
def test_stress_after_the_arrays_changed(precision, mode):
    import paper_1712_07739_gb300 as gb

    C = synth.isotropic_voigt(1.0, 0.3) if mode == "iso" else synth.cubic_voigt()
    f = gb.FMM(p=3, levels=3, precision=precision, h_mode=mode, circle_q=12).set_material(C)
    net = [torch.tensor(a, device="cuda") for a in synth.polygon_loops(n_segs=120, n_loops=6, seed=2)]
    x = torch.tensor(np.random.default_rng(1).uniform(0.2, 0.8, (200, 3)), device="cuda")
    f.build(*net)
    want = f.stress(x).cpu().numpy()
    net[0].mul_(1.5).add_(0.1)
    net[2].mul_(-3.0)
    assert np.array_equal(f.stress(x).cpu().numpy(), want)
