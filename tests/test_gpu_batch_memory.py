"""Device memory of an ensemble: what a pass only works in is shared by the networks that run one
after the other on a stream, so a network beyond the first eight adds its own tree and cell values."""
import numpy as np
import pytest

from paper_1712_07739_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_memory_per_network():
    import paper_1712_07739_gb300 as gb

    n, p, L = 20, 6, 5
    b = gb.Batch(n, p=p, levels=L, circle_q=16).set_material(synth.cubic_voigt())
    nets = [[torch.tensor(a, device="cuda") for a in synth.polygon_loops(n_segs=1000, n_loops=20, seed=k)]
            for k in range(n)]
    for k in range(8):
        b.build(k, *nets[k])
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for k in range(8, n):
        b.build(k, *nets[k])
    torch.cuda.synchronize()
    each = (before - torch.cuda.mem_get_info()[0]) / (n - 8)
    cells = (8 ** L - 1) // 7
    kp = (9 * p ** 3 + 63) // 64 * 64
    own = cells * p ** 3 * 15 * 4 + cells * kp * 2 * 2  # multipole and local values, packed operands
    print(f"{each / 2**20:.0f} MiB a network, {own / 2**20:.0f} of them cell values")
    assert each <= own + 16 * 2 ** 20
    # the networks' passes share scratch: each gives what it gives alone
    got = [f.clone() for f in b.nodal_forces()]
    for k in (0, 8, 16, n - 1):
        f = gb.FMM(p=p, levels=L, precision="mixed", h_mode="circle", circle_q=16).set_material(synth.cubic_voigt())
        f.build(*nets[k])
        want = f.nodal_forces()
        assert (got[k] - want).norm() <= 1e-12 * want.norm()
        f.close()
