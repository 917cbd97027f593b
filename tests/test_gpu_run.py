"""Many steps of a small lattice in one launch (k_run) against the same steps
as launches of their own (LBM_RUN=0): fields bit for bit where the per-node
arithmetic is the same (bounce-back and no solids), IBM and forces to rounding.
"""
import numpy as np
import pytest

from paper_1906_05445_gb300 import workloads as W

from .parity import rel_l2

pytestmark = pytest.mark.gpu

SPHERE = [W.Solid(W.SPHERE, (8.3, 9.1, 7.7), 3.2, omega=(0.002, 0.0, -0.001))]
GAP = [W.Solid(W.SPHERE, (6.2, 8.0, 8.0), 3.0), W.Solid(W.SPHERE, (13.4, 8.3, 7.9), 3.1)]
RING = [W.Solid(W.CYLINDER_Z, (16.3, 15.8, 0.0), 5.0, omega=(0.0, 0.0, 0.002)),
        W.Solid(W.CYLINDER_Z, (16.3, 15.8, 0.0), 13.0, fluid_inside=True)]


def _problem(lattice, shape, solids, scheme, precision, iters=1, collision=W.MRT):
    return W.Problem("run", lattice, *shape, 0.7, collision, precision, (1e-4, -2e-4, 0.0),
                     solids, scheme, 0, ibm_iters=iters)


# sizes: one node, odd rows (no vectors), fewer and more warps of nodes than
# blocks, more boundary-node groups than blocks (the 150^2 ring)
CASES = [(W.D3Q19, (1, 1, 1), [], W.NONE), (W.D3Q19, (5, 3, 2), [], W.NONE),
         (W.D3Q19, (20, 17, 16), SPHERE, W.BOUZIDI_QUAD), (W.D3Q19, (21, 17, 16), GAP, W.YU_QUAD),
         (W.D3Q19, (20, 17, 16), SPHERE, W.ZHAO_YONG), (W.D2Q9, (33, 32, 1), RING, W.BOUZIDI_LIN),
         (W.D2Q9, (64, 48, 1), RING, W.BB)]


def _step(p, monkeypatch, run, steps):
    import oracle as O
    from paper_1906_05445_gb300 import lbm
    monkeypatch.setenv("LBM_RUN", run)
    g = lbm.Lattice.from_problem(p)
    _, w = O.lattice(p.lattice)
    g.set_f(w.reshape((-1, 1, 1, 1)) * (1 + W.population_noise(
        p.Q, (p.nz if p.lattice == W.D3Q19 else 1, p.ny, p.nx), 4, 0.02)))
    for k in steps:
        g.step(k)
    f = g.get_f()
    u = g.velocity()
    hist = [g.force_history(s) for s in range(len(p.solids))]
    mask = g.solid_mask()
    g.sync()
    g.close()
    return f, u, hist, mask


@pytest.mark.parametrize("precision", [W.FP64, W.FP32, W.FP32_BF16, W.FP32_FP16])
@pytest.mark.parametrize("lattice,shape,solids,scheme", CASES)
def test_run_equals_launches(monkeypatch, lattice, shape, solids, scheme, precision):
    p = _problem(lattice, shape, solids, scheme, precision,
                 collision=W.BGK if lattice == W.D2Q9 else W.MRT)
    a = _step(p, monkeypatch, "0", (1, 2, 5))
    b = _step(p, monkeypatch, "1", (1, 2, 5))
    assert np.array_equal(a[0], b[0])
    for x, y in zip(a[2], b[2]):
        # FP64 sums of the same parts in another order: N 2^-53 of their size
        assert x.shape == y.shape and np.abs(x - y).max() <= 1e-12 * max(1.0, np.abs(x).max())


@pytest.mark.parametrize("iters", [1, 2, 5])
@pytest.mark.parametrize("precision,tol", [(W.FP64, 1e-13), (W.FP32, 2e-6)])
@pytest.mark.parametrize("lattice,shape,solids", [(W.D3Q19, (20, 17, 16), SPHERE),
                                                  (W.D3Q19, (24, 16, 16), GAP),
                                                  (W.D2Q9, (33, 32, 1), RING)])
def test_ibm_tables_equal_scattering(monkeypatch, lattice, shape, solids, precision, tol, iters):
    """The markers' tables (in k_run and by launches) against the scattering
    kernels: the same sums in another order, a few hundred roundings deep."""
    p = _problem(lattice, shape, solids, W.IBM, precision, iters)
    monkeypatch.setenv("LBM_IBM_TABLES", "0")
    a = _step(p, monkeypatch, "0", (1, 7))
    monkeypatch.setenv("LBM_IBM_TABLES", "1")
    for run in ("0", "1"):
        b = _step(p, monkeypatch, run, (1, 7))
        assert rel_l2(b[1], a[1], a[3]) <= tol
        for x, y in zip(a[2], b[2]):
            assert np.abs(x - y).max() <= 20 * tol * np.abs(x).max()
