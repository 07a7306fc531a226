"""Forces and stress in any unit of the moduli.

The kernel is homogeneous of degree one in the stiffness and every rounding in the passes scales
by the unit when that is a power of two, so results divided by the unit repeat those at unit one
but for FP32 range: bar 1e-6.  The units are near 1e-9, 1e5 (MPa) and 1e11 (Pa); a mixed pass that
forms a power of the moduli beyond the third in FP32 leaves its range at the outer two."""
import numpy as np
import pytest

from paper_1712_07739_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MEDIA = {"iso": synth.isotropic_voigt(1.0, 0.3), "cubic": synth.cubic_voigt(),
         "soft": synth.cubic_voigt(2.37, 1.11, 0.3),
         "turned": synth.rotated_voigt(synth.cubic_voigt(), synth.rotation())}
UNITS = [2.0 ** -30, 2.0 ** 17, 2.0 ** 37]


def _run(medium, unit, precision, mode, tol=None):
    import paper_1712_07739_gb300 as gb

    f = gb.FMM(p=4, levels=4, precision=precision, h_mode=mode, circle_q=17).set_material(MEDIA[medium] * unit)
    if mode == "mlp":
        rng = np.random.default_rng(3)
        theta = rng.normal(scale=0.08, size=gb.MLP_PARAMS).astype(np.float32)
        f.mlp_set(theta, rng.uniform(0.02, 0.08, 27).astype(np.float32) / np.float32(unit))
        f.mlp_calibrate(tol)
    nodes, segs, b = synth.polygon_loops(n_segs=400, n_loops=20, seed=8)
    f.build(*(torch.tensor(a, device="cuda") for a in (nodes, segs, b)))
    x = np.random.default_rng(4).uniform(nodes.min(0), nodes.max(0), (300, 3))
    out = [f.nodal_forces().cpu().numpy() / unit, f.stress(torch.tensor(x, device="cuda")).cpu().numpy() / unit]
    assert f.device_status() == 0
    f.close()
    return out


def _same(a, b):
    for x, y in zip(a, b):
        assert np.isfinite(x).all()
        assert np.linalg.norm(x - y) <= 1e-6 * np.linalg.norm(y), np.linalg.norm(x - y) / np.linalg.norm(y)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("medium", list(MEDIA))
def test_plain_rule(medium, precision):
    mode = "iso" if medium == "iso" else "circle"
    base = _run(medium, 1.0, precision, mode)
    for unit in UNITS:
        _same(_run(medium, unit, precision, mode), base)


@pytest.mark.parametrize("tol", [1e-30, 1e30])  # every bin on the plain rule; every bin on the network
@pytest.mark.parametrize("medium", ["cubic", "turned"])
def test_learned(medium, tol):
    base = _run(medium, 1.0, "mixed", "mlp", tol)
    for unit in UNITS:
        _same(_run(medium, unit, "mixed", "mlp", tol), base)
