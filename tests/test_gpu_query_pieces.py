"""Large fields into page-locked memory are computed and copied in pieces of
nodes: the same values as in one piece, for any place of the solids, and on
lattices of any size."""
import ctypes as C

import numpy as np
import pytest

from paper_1906_05445_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _pinned(n):
    import torch
    return torch.full((n,), -7.0, dtype=torch.float64).pin_memory().numpy()


@pytest.mark.parametrize("scheme", [W.BOUZIDI_QUAD, W.IBM])
@pytest.mark.parametrize("shape,centre", [((121, 80, 61), (60.2, 41.1, 30.4)),   # amid the pieces
                                          ((96, 96, 48), (1.3, 95.2, 0.4)),       # round the box's corner
                                          ((9, 11, 7001), (4.2, 5.1, 3500.3))])
def test_pieces_equal_one_copy(shape, centre, scheme):
    from paper_1906_05445_gb300 import lbm
    p = W.Problem("pieces", W.D3Q19, *shape, 0.7, W.MRT, W.FP64, (1e-4, -2e-4, 0.0),
                  [W.Solid(W.SPHERE, centre, 3.4)], scheme, 0)
    g = lbm.Lattice.from_problem(p)
    g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
    g.step(3)
    for fn, comps in ((lbm.lbm_get_density, 1), (lbm.lbm_get_velocity, 3),
                      (lbm.lbm_get_strain_rate, 6), (lbm.lbm_get_stress, 6),
                      (lbm.lbm_get_dissipation, 1), (lbm.lbm_get_distributions, 19)):
        one, pieces = np.full(comps * g.N, -7.0), _pinned(comps * g.N)
        for out in (one, pieces):
            assert fn(g.h, out.ctypes.data_as(C.POINTER(C.c_double)), out.size) == 0
        assert np.array_equal(one, pieces)
    g.close()


def test_page_locked_query_of_2_28_nodes():
    """Components of 2^31 bytes: more than the pitch of a 2D copy can be."""
    from paper_1906_05445_gb300 import lbm
    n = 1 << 14
    g = lbm.Lattice(W.D2Q9, n, n, 1, 0.7, precision=W.FP32_FP16)
    g.step(1)
    out = _pinned(2 * n * n)
    assert lbm.lbm_get_velocity(g.h, out.ctypes.data_as(C.POINTER(C.c_double)), out.size) == 0
    assert out.min() == 0.0 == out.max()
    g.close()
