"""The markers' tables of IBM solids at rest (rows of markers per band node,
coupled markers per marker), found through cells of markers, against the
scattering kernels: a missing or doubled entry would change the forces at once."""
import numpy as np
import pytest

from paper_1906_05445_gb300 import workloads as W

from .parity import rel_l2

pytestmark = pytest.mark.gpu

# smallest axes, cells that do not divide an axis, solids across every face and
# corner of the box, two solids whose stencils meet, cylinders, many markers per cell
CASES = [(W.D3Q19, (8, 9, 11), [W.Solid(W.SPHERE, (0.3, 8.6, 5.2), 2.2)], 1.0),
         (W.D3Q19, (13, 10, 8), [W.Solid(W.SPHERE, (12.7, 0.1, 7.9), 1.7)], 4.0),
         (W.D3Q19, (26, 19, 17), [W.Solid(W.SPHERE, (7.2, 8.0, 8.0), 3.9),
                                  W.Solid(W.SPHERE, (16.4, 8.3, 7.9), 4.1)], 1.0),
         (W.D3Q19, (21, 22, 9), [W.Solid(W.CYLINDER_Z, (20.6, 21.7, 0.0), 5.0)], 1.0),
         (W.D2Q9, (8, 8, 1), [W.Solid(W.CYLINDER_Z, (7.8, 0.4, 0.0), 2.0)], 1.0),
         (W.D2Q9, (75, 61, 1), [W.Solid(W.CYLINDER_Z, (30.3, 60.9, 0.0), 17.0)], 6.0)]


def _run(p, monkeypatch, tables):
    from paper_1906_05445_gb300 import lbm
    monkeypatch.setenv("LBM_IBM_TABLES", tables)
    g = lbm.Lattice.from_problem(p)
    g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
    g.step(4)
    out = [(g.velocity(), g.solid_mask(), g.force_torque(0))]
    # the next geometry in the tables' memory, smaller and larger
    for density in (0.5, 1.5 * p.marker_density):
        g.set_scheme(W.IBM, p.ibm_iters, 0.0, density)
        g.set_solid_motion(0, centre=tuple(c + 0.37 for c in p.solids[0].centre))
        g.step(3)
        out.append((g.velocity(), g.solid_mask(), g.force_torque(0)))
    g.close()
    return out


@pytest.mark.parametrize("iters", [1, 4])
@pytest.mark.parametrize("precision,tol", [(W.FP64, 1e-13), (W.FP32, 2e-6)])
@pytest.mark.parametrize("lattice,shape,solids,density", CASES)
def test_tables_equal_scattering(monkeypatch, lattice, shape, solids, density, precision, tol, iters):
    """The same sums in another order, a few hundred roundings deep."""
    p = W.Problem("tables", lattice, *shape, 0.7, W.MRT, precision, (1e-4, -2e-4, 0.0), solids,
                  W.IBM, 0, ibm_iters=iters, marker_density=density)
    for a, b in zip(_run(p, monkeypatch, "0"), _run(p, monkeypatch, "1")):
        assert rel_l2(b[0], a[0], a[1]) <= tol
        assert np.abs(a[2][0] - b[2][0]).max() <= 20 * tol * np.abs(a[2][0]).max()


def test_tables_keep_their_memory():
    """Rebuilding the geometry over and over does not add to the lattice's memory."""
    from paper_1906_05445_gb300 import lbm
    p = W.fixed_sphere(24, 3.1, seed=1, tau=0.7, g=2e-5, scheme=W.IBM, precision=W.FP32).with_(ibm_iters=3)
    sizes = {}
    for tables in (False, True):
        with pytest.MonkeyPatch.context() as mp:
            mp.setenv("LBM_IBM_TABLES", str(int(tables)))
            g = lbm.Lattice.from_problem(p)
            g.init_equilibrium()
            held = []
            for k in range(8):
                g.set_solid_motion(0, centre=(12.0 + 0.1 * k, 12.0, 12.0))
                g.step(2)
                held.append(g.info().device_bytes)
            g.close()
        sizes[tables] = np.array(held)
    extra = sizes[True] - sizes[False]
    assert extra[0] > 0 and extra[-1] <= 1.3 * extra[0]


@pytest.mark.parametrize("precision", [W.FP64, W.FP32])
@pytest.mark.parametrize("iters", [1, 3])
def test_new_rotation_keeps_the_geometry(precision, iters):
    """A new angular velocity of an IBM solid at rest changes the markers' desired
    velocities only: the same fields as after a rebuild of everything."""
    from paper_1906_05445_gb300 import lbm
    p = W.Problem("turn", W.D3Q19, 26, 19, 17, 0.7, W.MRT, precision, (1e-4, -2e-4, 0.0),
                  CASES[2][2], W.IBM, 0, ibm_iters=iters)
    out = []
    for rebuild in (False, True):
        g = lbm.Lattice.from_problem(p)
        g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
        g.step(3)
        for k in range(3):
            n0 = g.info().kernel_launches
            g.set_solid_motion(1, omega=(1e-3, 0.0, 2e-3 * k), velocity=(0.0, 0.0, 0.0))
            if rebuild:
                g.set_scheme(W.IBM, iters)
            g.step(2)
            assert (g.info().kernel_launches - n0 <= 2) != rebuild
        out.append((g.get_f(), g.force_torque(1)))
        g.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.abs(out[0][1][1] - out[1][1][1]).max() <= 1e-12
