"""The work that the roofline credits to the pair kernel (bench.near_work), per mode (CPU)."""
import os
import sys

import pytest

from paper_1712_07739_gb300 import synth

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

WORK = {"near_pairs": 1000, "points": 10}


def _wl(**kw):
    return dict(dict(p=5, circle_q=17, h_mode="circle", precision="mixed", C=synth.cubic_voigt), **kw)


def _turned():
    return synth.rotated_voigt(synth.cubic_voigt(), synth.rotation())


@pytest.mark.parametrize("wl,madds", [
    (_wl(), 39 * 8 + 430),                                      # 8 pairs of circle points, moments, cubic
    (_wl(precision="fp64"), 39 * 8 + 430),
    (_wl(circle_q=16), 39 * 7 + 430),
    (_wl(C=_turned), 132 * 17 + 190),                           # point by point
    (_wl(C=_turned, precision="fp64"), 39 * 8 + 850),           # moments, any medium
    (_wl(h_mode="iso", C=lambda: synth.isotropic_voigt(1.0, 0.3)), 2 * 43 + 30),
    (_wl(h_mode="mlp"), 108 + 220),
])
def test_near_work(wl, madds):
    flops, kernel = bench.near_work(wl, WORK)
    assert kernel == "k_near_pairs"
    # a pair once for both directions, a multiply-add as two; L2P per point
    assert flops == 500 * 2 * madds + 10 * (12 * 5 ** 3 + 30 * 5)


@pytest.mark.parametrize("wl,described", [(_wl(circle_q=16), True), (_wl(circle_q=16, precision="fp64"), False),
                                          (_wl(circle_q=16, h_mode="iso"), False), (_wl(circle_q=20), False)])
def test_traffic_only_where_a_capture_describes_it(wl, described):
    peaks = {"fp64_tflops": 1.0, "fp32_tflops": 80.0, "source": "test"}
    r = bench.roofline_of(wl, dict(WORK, m2l_pairs=1), 1.0, 2.0, 0, peaks)
    assert (r["traffic"] is not None) == described
