"""The grouped collision (collide_two_rate) of 16-bit storage: the packed pair
kernels and the node-by-node kernels give the same bits.
"""
import numpy as np
import pytest

from paper_1906_05445_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (lattice, shape, collision)
CASES = [(W.D3Q19, (12, 10, 8), W.MRT), (W.D3Q19, (40, 5, 3), W.BGK),
         (W.D2Q9, (24, 18, 1), W.MRT), (W.D2Q9, (72, 7, 1), W.BGK)]


def _run(monkeypatch, lattice, shape, collision, precision, packed, steps, g=(1e-4, -2e-4, 3e-4)):
    import oracle as O
    from paper_1906_05445_gb300 import lbm
    monkeypatch.setenv("LBM_VEC_PACKED", packed)
    nx, ny, nz = shape
    lat = lbm.Lattice(lattice, nx, ny, nz, 0.62, collision, precision, g)
    _, w = O.lattice(lattice)
    f0 = w.reshape((-1, 1, 1, 1)) * (1 + W.population_noise(len(w), (nz, ny, nx), 5, 0.05))
    lat.set_f(f0)
    lat.step(steps)
    f = lat.get_f()
    lat.close()
    return f


@pytest.mark.parametrize("precision", [W.FP32_BF16, W.FP32_FP16])
@pytest.mark.parametrize("lattice,shape,collision", CASES)
def test_packed_equals_node_by_node(monkeypatch, lattice, shape, collision, precision):
    a, b = (_run(monkeypatch, lattice, shape, collision, precision, p, 3) for p in ("0", "1"))
    assert np.array_equal(a, b)
