"""Where the multi-step launch of small lattices (k_run) meets the rest of the
library: geometry changed between launches, the ring of force records, captures,
long calls, refused launches, few and many blocks, lattices on several streams and
in batches, missing memory.  Compared with the same steps as launches of their own
(LBM_RUN=0).
"""
import numpy as np
import pytest

from paper_1906_05445_gb300 import workloads as W

from .parity import rel_l2

pytestmark = pytest.mark.gpu

DISC = [W.Solid(W.CYLINDER_Z, (15.7, 16.2, 0.0), 6.0, omega=(0.0, 0.0, 0.002))]


def _disc(precision, iters=1, scheme=W.IBM):
    return W.Problem("disc", W.D2Q9, 33, 32, 1, 0.7, W.MRT, precision, (1e-4, -2e-4, 0.0),
                     DISC, scheme, 0, ibm_iters=iters)


def _poison():
    """Leave small blocks of device memory that the next allocations may reuse
    full of NaN: the populations of lattices that held nothing else."""
    from paper_1906_05445_gb300 import lbm
    lats = []
    for n in [4, 8, 12, 16, 24] * 16:
        g = lbm.Lattice(W.D2Q9, n, n, 1, 0.7, precision=W.FP32)
        g.set_f(np.full((9, 1, n, n), np.nan))
        lats.append(g)
    for g in lats:
        g.close()


@pytest.mark.parametrize("iters", [1, 3])
@pytest.mark.parametrize("precision,tol", [(W.FP64, 1e-13), (W.FP32, 2e-6)])
def test_markers_changed_between_launches_2d(monkeypatch, precision, tol, iters):
    """New IBM tables straight into a multi-step launch, without an initial
    collision: the unused z component of the markers' forces reads as zero.
    Both runs sum the same few hundred terms in another order."""
    from paper_1906_05445_gb300 import lbm
    out = []
    for run in ("0", "1"):
        monkeypatch.setenv("LBM_RUN", run)
        g = lbm.Lattice.from_problem(_disc(precision, iters))
        g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
        g.step(4)
        # more markers: larger tables, in memory that held something else
        g.set_scheme(W.IBM, iters, 0.0, 6.0)
        g.set_solid_motion(0, centre=(15.9, 16.1, 0.0), omega=(0.0, 0.0, 0.001))
        _poison()
        g.step(9)
        out.append((g.velocity(), g.solid_mask(), g.force_torque(0)))
        g.close()
    assert np.isfinite(out[1][0]).all()
    assert rel_l2(out[1][0], out[0][0], out[0][1]) <= tol
    for a, b in zip(out[0][2], out[1][2]):
        assert np.abs(a - b).max() <= 20 * tol * np.abs(out[0][2][0]).max()


def test_whole_force_history_of_a_full_ring(monkeypatch):
    """Once more steps ran than records are kept, the history still holds the
    last 4096 steps, the oldest included."""
    from paper_1906_05445_gb300 import lbm
    hist = []
    for run in ("0", "1"):
        monkeypatch.setenv("LBM_RUN", run)
        g = lbm.Lattice.from_problem(_disc(W.FP64, scheme=W.BOUZIDI_QUAD))
        g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
        g.step(2100)
        g.step(2110)
        hist.append(g.force_history(0))
        g.close()
    assert hist[0].shape == hist[1].shape == (4096, 6)
    # FP64 sums of the same parts in another order
    assert np.abs(hist[0] - hist[1]).max() <= 1e-12 * max(1.0, np.abs(hist[0]).max())
    assert np.abs(hist[1][0, :2]).min() > 1e-8


def test_captured_launch_clears_no_record_by_itself(monkeypatch):
    """Steps captured into a graph that is never launched leave every record
    as it was: the next launch clears its own first one."""
    import torch
    from paper_1906_05445_gb300 import lbm
    out = []
    for run in ("0", "1"):
        monkeypatch.setenv("LBM_RUN", run)
        s = torch.cuda.Stream()
        g = lbm.Lattice.from_problem(_disc(W.FP64, scheme=W.BOUZIDI_QUAD), stream=s.cuda_stream)
        g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
        g.step(4200)  # every slot of the ring holds a record
        g.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
            g.step(2)
        g.step(3)
        out.append(g.force_history(0, 3))
        g.close()
        del graph
    assert np.abs(out[0] - out[1]).max() <= 1e-12 * max(1.0, np.abs(out[0]).max())


@pytest.mark.parametrize("scheme", [W.BOUZIDI_QUAD, W.IBM])
def test_long_calls_run_in_launches_of_bounded_length(monkeypatch, scheme):
    """A call of many steps is split: 600 steps are three launches, with the
    results of the same steps in short calls."""
    from paper_1906_05445_gb300 import lbm
    monkeypatch.setenv("LBM_RUN", "1")
    out = []
    for calls in ((600,), (100,) * 6):
        g = lbm.Lattice.from_problem(_disc(W.FP32, 2, scheme=scheme))
        g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
        g.step(2)
        n0 = g.info().kernel_launches
        for k in calls:
            g.step(k)
        out.append((g.info().kernel_launches - n0, g.get_f(), g.force_history(0)))
        g.close()
    assert out[0][0] == 3 and out[1][0] == 6
    assert np.array_equal(out[0][1], out[1][1])
    # FP64 sums of the same parts in another order
    assert np.abs(out[0][2] - out[1][2]).max() <= 1e-12 * max(1.0, np.abs(out[0][2]).max())


@pytest.mark.parametrize("scheme", [W.BOUZIDI_QUAD, W.IBM])
def test_refused_launch_steps_with_launches(monkeypatch, scheme):
    """More blocks than the device holds at once (LBM_RUN_SMS above its SMs, as
    on a stream with fewer SMs): the runtime refuses the cooperative launch on
    the host, and the lattice steps with launches of its own, alone and in a
    batch."""
    from paper_1906_05445_gb300 import lbm
    p = _disc(W.FP64, scheme=scheme).with_(nx=192, ny=190)
    out = []
    for run, sms in (("0", ""), ("1", "1200")):
        monkeypatch.setenv("LBM_RUN", run)
        if sms:
            monkeypatch.setenv("LBM_RUN_SMS", sms)
        lats = [lbm.Lattice.from_problem(p) for _ in range(2)]
        for g in lats:
            g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
        b = lbm.Batch(lats, autotune=False)
        b.step(6)
        b.close()
        lats[0].step(5)
        n0 = lats[0].info().kernel_launches
        lats[0].step(3)
        assert lats[0].info().kernel_launches - n0 >= 6
        out.append([(g.get_f(), g.force_torque(0)) for g in lats])
        for g in lats:
            g.sync()
            g.close()
    for a, b in zip(*out):
        assert np.array_equal(a[0], b[0])
        for x, y in zip(a[1], b[1]):
            assert np.abs(x - y).max() <= 1e-12 * max(1.0, np.abs(x).max())


SPHERE = [W.Solid(W.SPHERE, (8.3, 9.1, 7.7), 3.2, omega=(0.002, 0.0, -0.001))]
ROUTES = [("0", ""), ("1", ""), ("1", "1"), ("1", "5"), ("1", "40")]


def _routes(monkeypatch, lattice, shape, solids, precision, scheme, iters=1, density=1.0):
    """Launches, and multi-step launches on one block (every boundary node and
    marker of the lattice in turn), a few and many blocks (one group of boundary
    nodes per block, one marker per warp)."""
    from paper_1906_05445_gb300 import lbm
    p = W.Problem("routes", lattice, *shape, 0.7, W.MRT, precision, (1e-4, -2e-4, 0.0), solids,
                  scheme, 0, ibm_iters=iters, marker_density=density)
    out = []
    for run, sms in ROUTES:
        monkeypatch.setenv("LBM_RUN", run)
        if sms:
            monkeypatch.setenv("LBM_RUN_SMS", sms)
        g = lbm.Lattice.from_problem(p)
        g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
        g.step(1)
        g.step(6)
        out.append((g.get_f(), g.velocity(), g.force_history(0), g.solid_mask()))
        g.sync()
        g.close()
    return out


@pytest.mark.parametrize("precision", [W.FP64, W.FP32, W.FP32_BF16, W.FP32_FP16])
@pytest.mark.parametrize("scheme", [W.BOUZIDI_QUAD, W.ZHAO_YONG])
@pytest.mark.parametrize("lattice,shape,solids", [(W.D3Q19, (20, 17, 16), SPHERE),
                                                  (W.D2Q9, (33, 32, 1), DISC)])
def test_blocks_of_a_launch_do_not_show(monkeypatch, lattice, shape, solids, precision, scheme):
    a, *rest = _routes(monkeypatch, lattice, shape, solids, precision, scheme)
    for b in rest:
        assert np.array_equal(a[0], b[0])
        # FP64 sums of the same parts in another order
        assert np.abs(a[2] - b[2]).max() <= 1e-12 * max(1.0, np.abs(a[2]).max())


@pytest.mark.parametrize("precision,tol", [(W.FP64, 1e-13), (W.FP32, 2e-6)])
@pytest.mark.parametrize("iters,density", [(1, 1.0), (5, 1.0), (2, 5.0)])
@pytest.mark.parametrize("lattice,shape,solids", [(W.D3Q19, (20, 17, 16), SPHERE),
                                                  (W.D2Q9, (33, 32, 1), DISC)])
def test_blocks_of_an_ibm_launch(monkeypatch, lattice, shape, solids, precision, tol, iters,
                                 density):
    """At density 5 a node's row holds more markers than its group has threads
    for.  The same sums in another order, a few hundred roundings deep."""
    a, *rest = _routes(monkeypatch, lattice, shape, solids, precision, W.IBM, iters, density)
    for b in rest:
        assert rel_l2(b[1], a[1], a[3]) <= tol
        assert np.abs(a[2] - b[2]).max() <= 20 * tol * np.abs(a[2]).max()


def test_lattices_on_streams_of_their_own_share_the_sms(monkeypatch):
    """Stepped in turn, lattices on streams of their own take a share of the SMs
    each, and launches of their own where the share is too small for them; one
    stepped alone has them all again.  The fields do not depend on it."""
    import torch
    from paper_1906_05445_gb300 import lbm
    p = W.Problem("share", W.D3Q19, 58, 58, 58, 0.7, W.MRT, W.FP32, (1e-4, -2e-4, 0.0), SPHERE,
                  W.BOUZIDI_QUAD, 0)
    monkeypatch.setenv("LBM_RUN", "0")
    ref = lbm.Lattice.from_problem(p)
    ref.init_equilibrium(1.0, (0.01, 0.005, 0.0))
    ref.step(16)
    monkeypatch.setenv("LBM_RUN", "1")
    streams = [torch.cuda.Stream() for _ in range(3)]
    lats = [lbm.Lattice.from_problem(p, stream=s.cuda_stream) for s in streams]

    def launches(g, k):
        n0 = g.info().kernel_launches
        g.step(k)
        return g.info().kernel_launches - n0

    for g in lats:
        g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
        g.step(1)
    assert all(launches(g, 3) > 1 for g in lats)  # a third of the SMs each
    assert launches(lats[0], 2) > 1               # the others stepped since
    assert launches(lats[0], 2) == 1              # alone
    assert launches(lats[1], 2) > 1               # after both others
    assert launches(lats[0], 2) == 1              # beside one other: half
    assert launches(lats[1], 2) == 1
    lats[0].step(6)
    lats[1].step(8)
    lats[2].step(12)
    for g in lats:
        assert np.array_equal(g.get_f(), ref.get_f())
        g.close()
    ref.close()


def test_batch_takes_one_route_for_all(monkeypatch):
    """A batch of small lattices runs in multi-step launches; with a lattice among
    them that does not (here: a moving solid), all step by graph replays or
    launches.  Both give the populations of the lattices stepped alone."""
    from paper_1906_05445_gb300 import lbm
    monkeypatch.setenv("LBM_RUN", "1")
    small = [W.Problem("b", W.D3Q19, n, 17, 16, 0.7, W.MRT, W.FP32, (1e-4, -2e-4, 0.0), SPHERE,
                       W.BOUZIDI_QUAD, 0) for n in (20, 24, 31)]
    moving = W.translating_sphere(36, 20, 20, 4.3, seed=23, u=0.05, tau=0.7,
                                  scheme=W.BOUZIDI_QUAD, precision=W.FP32)
    for extra, launches in (([], [1, 2]), ([moving], [4, 7])):
        alone = [lbm.Lattice.from_problem(p) for p in small + extra]
        mixed = [lbm.Lattice.from_problem(p) for p in small + extra]
        b = lbm.Batch(mixed, autotune=False)
        for k, n in zip((9, 6), launches):
            b.step(k)
            for g in alone:
                g.step(k)
            assert b.info(0)[2] == n
        for a, m in zip(alone, mixed):
            assert np.array_equal(a.get_f(), m.get_f())
            assert m.info().steps == 15
        b.close()
        for g in alone + mixed:
            g.close()


@pytest.mark.parametrize("iters", [1, 3])
def test_no_memory_for_the_tables(monkeypatch, iters):
    """Where the markers' tables find no memory, the lattice steps without them,
    as with LBM_IBM_TABLES=0."""
    from paper_1906_05445_gb300 import lbm
    p = _disc(W.FP64, iters)

    def run(allowed):
        lbm.debug_fail_allocations_after(allowed)
        g = None
        try:
            g = lbm.Lattice.from_problem(p)
            g.init_equilibrium(1.0, (0.01, 0.005, 0.0))
            g.step(5)
            lbm.debug_fail_allocations_after(-1)
            return g.velocity(), g.solid_mask(), g.force_torque(0)
        except lbm.LbmError as e:
            assert "OOM" in str(e)
        finally:
            lbm.debug_fail_allocations_after(-1)
            if g is not None:
                g.close()

    monkeypatch.setenv("LBM_IBM_TABLES", "0")
    need = next(k for k in range(200) if run(k) is not None)
    ref = run(need)
    monkeypatch.setenv("LBM_IBM_TABLES", "1")
    assert run(need - 1) is None
    for extra in (0, 1, 4, 9):
        got = run(need + extra)
        assert rel_l2(got[0], ref[0], ref[1]) <= 1e-13
        assert np.abs(got[2][0] - ref[2][0]).max() <= 2e-12 * np.abs(ref[2][0]).max()


def test_batch_reports_the_boundary_kernels_width():
    from paper_1906_05445_gb300 import lbm
    lats = [lbm.Lattice.from_problem(_disc(W.FP32, scheme=s)) for s in (W.BOUZIDI_QUAD, W.IBM)]
    b = lbm.Batch(lats, autotune=False)
    b.step(2)
    assert [b.info(i)[1] for i in range(2)] == [128, 64]
    b.close()
    for g in lats:
        g.close()
