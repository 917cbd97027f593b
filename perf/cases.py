"""The work that users of the library have it do, as measurable cases.

A case is a dict of plain values; ``prepare`` makes the lattices and their
inputs on the GPU, ``run`` is one pass through the public entry points,
``work`` says what a pass cannot do without, and ``exact`` computes the same
outputs with plain torch in 64 bits (its own collision, streaming, bounce-back,
immersed boundary, domain faces and solid motion; none of the library's code).

Outputs are the whole post-collision populations (the library's own device
buffer) beside the sampled force, torque and motion.  Values that a lattice
computes in 32 bits but hands out in FP64 containers (force, torque, residual)
are returned in the type of the lattice's storage.
"""
import math

import numpy as np
import torch

from paper_1906_05445_gb300 import lbm
from paper_1906_05445_gb300 import workloads as W

PREC = {"fp64": W.FP64, "fp32": W.FP32, "bf16": W.FP32_BF16, "fp16": W.FP32_FP16}
SCHEME = {"bouzidi_lin": W.BOUZIDI_LIN, "bouzidi_quad": W.BOUZIDI_QUAD, "ibm": W.IBM,
          "zhao_yong": W.ZHAO_YONG}
BYTES = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}
FLOPS = {2: 90.0, 3: 210.0}  # arithmetic of one node update (D2Q9, D3Q19)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the paper's circular Couette flow at its smallest: a few thousand
        # nodes, FP64, sampled every 100 steps -- launches and latency
        {"name": "couette_64_fp64", "kind": "couette", "n": 64, "precision": "fp64",
         "scheme": "bouzidi_lin", "steps": 100},
        # a served 2D solve (request sizes are any integer): one round of 200
        # steps between residual checks, odd edge, FP32
        {"name": "steady_301_fp32", "kind": "steady", "n": 301, "precision": "fp32",
         "scheme": "bouzidi_quad", "steps": 200},
        # the settling cylinder: closed channel, free solid moving on the
        # device, graph replays between samples of its position
        {"name": "settling_80x800_fp64", "kind": "settling", "d": 20, "precision": "fp64",
         "scheme": "bouzidi_quad", "steps": 40},
        # a small sphere under IBM with five forcing iterations (the paper's
        # n_it): a chain of short dependent kernels
        {"name": "sphere_48_ibm5_fp32", "kind": "sphere", "n": 48, "precision": "fp32",
         "scheme": "ibm", "iters": 5, "steps": 40},
        # the 128^3 sphere of the benchmark under bounce-back, drag sampled
        # every 20 steps
        {"name": "sphere_128_ibb_fp32", "kind": "sphere", "n": 128, "precision": "fp32",
         "scheme": "bouzidi_quad", "iters": 1, "steps": 20},
        # the benchmark itself: bounce-back and IBM lattices side by side on
        # their own streams, the force record of every step copied out
        {"name": "pair_128_fp32", "kind": "pair", "n": 128, "precision": "fp32", "steps": 20},
        # FP64, as the accuracy studies run it
        {"name": "sphere_96_fp64", "kind": "sphere", "n": 96, "precision": "fp64",
         "scheme": "bouzidi_quad", "iters": 1, "steps": 5},
        # 16-bit storage where it is accurate enough: IBM, FP16
        {"name": "sphere_160_ibm_fp16", "kind": "sphere", "n": 160, "precision": "fp16",
         "scheme": "ibm", "iters": 1, "steps": 10},
        # the translating sphere: geometry rebuilt and nodes refilled each step
        {"name": "moving_256x128x128_fp32", "kind": "moving", "nx": 256, "ny": 128, "nz": 128,
         "radius": 8.0, "precision": "fp32", "scheme": "bouzidi_quad", "steps": 10},
        # uniform flow past a sphere in the open box at the drag study's
        # finest grid: 48 M nodes, single-node bounce-back, every face open,
        # a slowly turning sphere
        {"name": "open_d24_fp32", "kind": "open", "d": 24, "precision": "fp32",
         "scheme": "zhao_yong", "steps": 4},
        # the grid-convergence batch: eight lattices of edges 24...64,
        # alternating bounce-back and IBM, graph replays
        {"name": "batch_8_fp32", "kind": "batch", "count": 8, "r_max": 8.0, "precision": "fp32",
         "steps": 40},
        # post-processing: velocity, strain rate and dissipation rate read
        # into page-locked host memory
        {"name": "fields_96_fp64", "kind": "fields", "n": 96, "precision": "fp64",
         "scheme": "bouzidi_quad"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["couette", "steady", "settling", "sphere", "sphere", "sphere", "pair",
                       "moving", "open", "batch", "fields"])
    if kind in ("couette", "steady"):
        return {"kind": kind, "n": _log(rng, 48, 512), "precision": rng.choice(["fp64", "fp32"]),
                "scheme": rng.choice(["bouzidi_lin", "bouzidi_quad"]),
                "steps": rng.randrange(50, 201)}
    if kind == "settling":
        return {"kind": kind, "d": rng.randrange(10, 25), "precision": "fp64",
                "scheme": "bouzidi_quad", "steps": rng.randrange(10, 61)}
    if kind == "sphere":
        prec = rng.choice(["fp32", "fp32", "fp64", "bf16", "fp16"])
        scheme = "ibm" if prec == "fp16" else rng.choice(["bouzidi_lin", "bouzidi_quad", "ibm"])
        return {"kind": kind, "n": _log(rng, 24, 96 if prec == "fp64" else 192), "precision": prec,
                "scheme": scheme, "iters": rng.choice([1, 1, 3, 5]) if scheme == "ibm" else 1,
                "steps": rng.randrange(2, 25)}
    if kind == "pair":
        return {"kind": kind, "n": _log(rng, 48, 144), "precision": "fp32",
                "steps": rng.randrange(5, 25)}
    if kind == "moving":
        return {"kind": kind, "nx": _log(rng, 64, 256), "ny": _log(rng, 48, 128),
                "nz": _log(rng, 48, 128), "radius": rng.choice([4.0, 6.0, 8.0]),
                "precision": rng.choice(["fp32", "fp32", "fp16"]), "scheme": "bouzidi_quad",
                "steps": rng.randrange(4, 13)}
    if kind == "open":
        return {"kind": kind, "d": rng.randrange(8, 17), "precision": "fp32",
                "scheme": rng.choice(["zhao_yong", "bouzidi_quad", "ibm"]),
                "steps": rng.randrange(2, 6)}
    if kind == "batch":
        return {"kind": kind, "count": rng.randrange(2, 11), "r_max": rng.choice([6.0, 8.0, 10.0]),
                "precision": "fp32", "steps": rng.randrange(10, 61)}
    return {"kind": "fields", "n": _log(rng, 24, 112), "precision": "fp64",
            "scheme": "bouzidi_quad"}


# ----------------------------------------------------------------- the inputs
def _problems(case, seed):
    """The lattices of a case, as workload problems (seeded geometry)."""
    rng = np.random.default_rng([1906, seed])
    kind = case["kind"]
    prec = PREC[case["precision"]]
    if kind in ("couette", "steady"):
        n = case["n"]
        c = (n / 2 + float(rng.random()), n / 2 + float(rng.random()))
        r1 = n / 6.4
        return [W.couette_2d(n, r1, 2.8 * r1, c, 0.01, float(rng.uniform(0.7, 0.9)),
                             SCHEME[case["scheme"]], 0, prec)]
    if kind == "settling":
        d = case["d"]
        x = 1.62 * d + float(rng.random())
        y = 30.0 * d + float(rng.random())
        p = W.Problem("settling", W.D2Q9, 4 * d, 40 * d, 1, 0.6, W.MRT, prec, (0.0, 0.0, 0.0),
                      [W.Solid(W.SPHERE, (x, y, 0.0), d / 2)], SCHEME[case["scheme"]], 0,
                      faces=(W.VELOCITY,) * 4 + (W.PERIODIC,) * 2,
                      u_face=((0.0, 0.0, 0.0),) * 6)
        return [p]
    s = int(rng.integers(1 << 30))
    if kind in ("sphere", "fields"):
        n = case["n"]
        return [W.fixed_sphere(n, 3.0 * n / 32.0, s, 0.6, 1e-6, SCHEME[case["scheme"]], prec,
                               W.MRT, 0, ibm_iters=case.get("iters", 1))]
    if kind == "pair":
        n = case["n"]
        return [W.fixed_sphere(n, 3.0 * n / 32.0, s, 0.6, 1e-6, sch, prec, W.MRT, 0)
                for sch in (W.BOUZIDI_QUAD, W.IBM)]
    if kind == "moving":
        return [W.translating_sphere(case["nx"], case["ny"], case["nz"], case["radius"], s,
                                     0.01, 0.6, SCHEME[case["scheme"]], prec, 0)]
    if kind == "open":
        p = W.open_sphere(D=float(case["d"]), re=20.0, nu=0.04, seed=s,
                          scheme=SCHEME[case["scheme"]], precision=prec)
        # the sphere turns slowly (a tenth of the stream's speed at its surface)
        b = p.solids[0]
        b.omega = tuple(0.1 * p.u_face[0][0] / b.radius * v for v in (0.2, -0.3, 1.0))
        return [p]
    ps = W.convergence_batch(case["count"], s, 0.8, 2.0, 3.0, case["r_max"])
    return [p.with_(precision=prec) for p in ps]


def _lattice(p):
    """(velocities [Q][3] in the library's direction order, weights)."""
    if p.lattice == W.D2Q9:
        e = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        return [v + (0,) for v in e], [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    e = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
         (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
         (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
    return e, [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _shape(p):
    return (p.nz if p.lattice == W.D3Q19 else 1, p.ny, p.nx)


def _initial(p, seed, k):
    """Deviations f_i - w_i of a smooth flow (a few Fourier modes, speeds of
    order 1e-2, density within 0.2%) as a list of FP64 tensors."""
    rng = np.random.default_rng([7, seed, k])
    e, w = _lattice(p)
    D = 2 if p.lattice == W.D2Q9 else 3
    nz, ny, nx = _shape(p)
    grid = [2 * math.pi * torch.arange(m, dtype=torch.float64, device="cuda") / m
            for m in (nz, ny, nx)]
    z, y, x = (grid[0].view(-1, 1, 1), grid[1].view(1, -1, 1), grid[2].view(1, 1, -1))
    u = []
    for c in range(4):
        v = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
        if c < D or c == 3:
            for _ in range(2):
                kz, ky, kx = (int(rng.integers(1, 3)) if D == 3 else 0, int(rng.integers(1, 3)),
                              int(rng.integers(1, 3)))
                v += float(rng.uniform(0.3, 1.0)) * torch.sin(
                    kx * x + ky * y + kz * z + float(rng.uniform(0, 2 * math.pi)))
        u.append(v * (0.01 if c < 3 else 0.001))
    return _feq(e, w, u[3], u[:3])


def _feq(e, w, drho, u):
    uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    out = []
    for ei, wi in zip(e, w):
        eu = _edot(ei, u)
        out.append(wi * (drho + 3 * eu + 4.5 * eu * eu - 1.5 * uu))
    return out


def _edot(ei, v):
    s = 0
    for c in range(3):
        if ei[c]:
            s = s + ei[c] * v[c]
    return s + 0 * v[0]


def _starts_uniform(case):
    return case["kind"] == "open"


class _Raw:
    """A library buffer for torch; the tensor keeps this object, and with it
    the lattice that owns the memory, alive."""

    def __init__(self, owner, ptr, count, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": (count,),
                                         "typestr": typestr, "version": 3}


class _State:
    """One lattice and the torch views of its two population buffers."""

    def __init__(self, p, stream=None):
        self.p = p
        self.lat = lbm.Lattice.from_problem(p, stream=stream)
        self.views = {}
        self.ptr, self.nbytes, self.stride = lbm.C.c_void_p(), lbm.C.c_size_t(), lbm.C.c_size_t()

    def f(self):
        """The current post-collision populations [Q][nodes], in place."""
        st = lbm.lbm_device_field(self.lat.h, 0, lbm.C.byref(self.ptr), lbm.C.byref(self.nbytes),
                                  lbm.C.byref(self.stride))
        if st != lbm.LBM_OK:
            raise RuntimeError("lbm_device_field")
        key = (self.ptr.value, self.stride.value)
        if key not in self.views:
            size = {W.FP64: 8, W.FP32: 4}.get(self.p.precision, 2)
            typ = {W.FP64: "<f8", W.FP32: "<f4", W.FP32_BF16: "<i2", W.FP32_FP16: "<f2"}
            t = torch.as_tensor(_Raw(self.lat, self.ptr.value, self.nbytes.value // size,
                                     typ[self.p.precision]), device="cuda")
            if self.p.precision == W.FP32_BF16:
                t = t.view(torch.bfloat16)
            self.views[key] = t.view(self.p.Q, self.stride.value)[:, :self.p.nodes]
        return self.views[key]

    def own(self, *values):
        """Host values in the type of the lattice's storage."""
        if self.p.precision == W.FP64:
            return list(values)
        if self.p.precision == W.FP32:
            return [np.asarray(v, dtype=np.float32) for v in values]
        t = torch.bfloat16 if self.p.precision == W.FP32_BF16 else torch.float16
        return [torch.as_tensor(v).to(t) for v in values]

    def start(self, case, seed, k):
        p, lat = self.p, self.lat
        if _starts_uniform(case):
            lat.init_equilibrium(1.0, p.u_face[0])
        else:
            _, w = _lattice(p)
            d = _initial(p, seed, k)
            f0 = torch.stack([di + wi for di, wi in zip(d, w)]).cpu().numpy()
            lat.set_f(f0)
        # nodes inside solids hold no populations: zero, not whatever the
        # fresh buffer contained
        f = self.f()
        solid = torch.from_numpy(lat.solid_mask().reshape(-1)).cuda()
        f[:, solid] = 0
        torch.cuda.synchronize()


def prepare(case, seed):
    kind = case["kind"]
    ps = _problems(case, seed)
    streams = [torch.cuda.Stream() if kind == "pair" else None for _ in ps]
    sts = [_State(p, s.cuda_stream if s else None) for p, s in zip(ps, streams)]
    state = {"case": dict(case), "lats": sts, "streams": streams}
    if kind == "settling":
        sts[0].lat.set_solid_dynamics(0, 1.03, _gravity(case))
    for k, s in enumerate(sts):
        s.start(case, seed, k)
    if kind in ("settling", "batch"):
        state["batch"] = lbm.Batch([s.lat for s in sts])
    if kind == "pair":
        state["rec"] = [torch.zeros((case["steps"], 6), dtype=torch.float64).pin_memory()
                        for _ in sts]
        state["rows"] = [[row for row in r.numpy()] for r in state["rec"]]
    if kind == "fields":
        sts[0].lat.step(2)
        n = ps[0].nodes
        state["host"] = [torch.zeros((c, n), dtype=torch.float64).pin_memory().numpy()
                         for c in (3, 6, 1)]
    return state


def _gravity(case):
    # settles at about a thousandth of a node per step
    return (0.0, -2e-4 * (20.0 / case["d"]) ** 2, 0.0)


# ------------------------------------------------------------------- one pass
def run(state):
    case, sts = state["case"], state["lats"]
    kind, n = case["kind"], case.get("steps", 0)
    s = sts[0]
    if kind in ("couette", "sphere", "moving", "open"):
        s.lat.step(n)
        F, T = s.own(*s.lat.force_torque(0))
        return {"f": s.f(), "force": F, "torque": T}
    if kind == "steady":
        steps, r = s.lat.run_to_steady(1e-30, n, n)
        return {"f": s.f(), "steps": steps, "residual": s.own(np.array([r]))[0]}
    if kind == "settling":
        state["batch"].step(n)
        U, Om = s.lat.solid_velocity(0)
        return {"f": s.f(), "centre": s.lat.solid_centre(0), "velocity": U, "omega": Om}
    if kind == "batch":
        state["batch"].step(n)
        out = {}
        for k, t in enumerate(sts):
            F, T = t.own(*t.lat.force_torque(0))
            out["lattice%02d" % k] = {"f": t.f(), "force": F, "torque": T}
        return out
    if kind == "pair":
        rows = state["rows"]
        a, b = sts[0].lat, sts[1].lat
        for k in range(n):
            a.step(1)
            a.copy_force_torque_async(rows[0][k])
            b.step(1)
            b.copy_force_torque_async(rows[1][k])
        a.sync()
        b.sync()
        return {"f_ibb": sts[0].f(), "f_ibm": sts[1].f(),
                "record_ibb": state["rec"][0].float(), "record_ibm": state["rec"][1].float()}
    h = state["host"]
    lat = s.lat
    lat.velocity(out=h[0])
    for fn, out in ((lbm.lbm_get_strain_rate, h[1]), (lbm.lbm_get_dissipation, h[2])):
        if fn(lat.h, out.ctypes.data_as(lbm.C.POINTER(lbm.C.c_double)), out.size) != lbm.LBM_OK:
            raise RuntimeError("field query")
    return {"velocity": h[0], "strain": h[1], "dissipation": h[2]}


def work(case):
    """Populations read once and written once per pass; the arithmetic of
    every node update."""
    b = f = 0.0
    for p in _problems(case, 0):
        D = 2 if p.lattice == W.D2Q9 else 3
        if case["kind"] == "fields":
            b += p.nodes * (p.Q * BYTES[case["precision"]] + 10 * 8.0)
            f += p.nodes * 150.0
        else:
            b += 2.0 * p.nodes * p.Q * BYTES[case["precision"]]
            f += p.nodes * FLOPS[D] * case["steps"]
    return {"bytes": b, "flops": f}


# ------------------------------------------------- the same, in 64-bit torch
class _Ref:
    """Collide-and-stream in FP64 torch: BGK or two-rate MRT with Guo forcing,
    interpolated bounce-back (linear and quadratic Bouzidi, Zhao-Yong),
    direct-forcing IBM, domain faces, prescribed and free solids."""

    def __init__(self, p, d0, uniform):
        self.p = p
        self.e, self.w = _lattice(p)
        self.Q = len(self.e)
        self.D = 2 if p.lattice == W.D2Q9 else 3
        self.opp = [self.e.index(tuple(-c for c in v)) for v in self.e]
        self.shape = _shape(p)
        self.len = [p.nx, p.ny, self.shape[0]]
        self.omega = 1.0 / p.tau
        self.sq = 1.0 / (0.5 + (3.0 / 16.0) / (p.tau - 0.5))
        self.mrt = p.collision == W.MRT
        self.ibm = p.scheme == W.IBM
        self.c = [list(s.centre) for s in p.solids]
        self.U = [list(s.velocity) for s in p.solids]
        self.Om = [list(s.omega) for s in p.solids]
        self.rho_p, self.grav = 0.0, (0.0, 0.0, 0.0)
        self.moving = any(any(s.velocity) for s in p.solids)
        if self.D == 2:
            for k in range(len(self.c)):
                self.c[k][2] = 0.0
        self.geometry()
        ns = ~self.solid
        f = [di if uniform else torch.where(ns, di, torch.zeros_like(di)) for di in d0]
        self.pre = [t.clone() for t in f] if p.scheme == W.ZHAO_YONG else None
        if p.faces is not None and W.CONVECTIVE in p.faces:
            self.keep_outlet(f, self.forces(f)[0])
        self.force = np.zeros((1, 6))
        F, rec = self.forces(f)
        if rec is not None:
            self.force = rec
        post = self.collide([t.clone() for t in f], F)
        self.post = [torch.where(ns, t, torch.zeros_like(t)) for t in post]
        self.other = f  # the buffer the next step writes into
        self.f = f      # the pre-collision state
        self.F = F

    # -- geometry at the current centres
    def coords(self):
        nz, ny, nx = self.shape
        a = [torch.arange(m, dtype=torch.float64, device="cuda") for m in (nx, ny, nz)]
        return a[0].view(1, 1, -1), a[1].view(1, -1, 1), a[2].view(-1, 1, 1)

    def rel(self, s, x, y, z):
        b, c = self.p.solids[s], self.c[s]
        flat = self.D == 2 or b.kind == W.CYLINDER_Z
        r = []
        for v, c0, m in ((x, c[0], self.p.nx), (y, c[1], self.p.ny)):
            d = v - c0
            r.append(d - m * torch.round(d / m))
        d = z - c[2]
        r.append(0 * d if flat else d - self.shape[0] * torch.round(d / self.shape[0]))
        return r

    def geometry(self):
        x, y, z = self.coords()
        sid = torch.zeros(self.shape, dtype=torch.int8, device="cuda")
        for s in reversed(range(len(self.p.solids))):
            r = self.rel(s, x, y, z)
            r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2]
            R2 = self.p.solids[s].radius ** 2
            sid[(r2 >= R2) if self.p.solids[s].fluid_inside else (r2 <= R2)] = s + 1
        self.sid = sid
        if self.ibm:
            self.solid = torch.zeros_like(sid, dtype=torch.bool)
            self.g_on = (sid == 0).double()
        else:
            self.solid = sid != 0
            self.g_on = 1.0
        self.links = []
        if self.ibm:
            return
        nx, ny, nz = self.len
        for i in range(1, self.Q):
            ei = self.e[i]
            behind = torch.roll(sid, (ei[2], ei[1], ei[0]), (0, 1, 2))  # the id at x - e_i
            n = torch.nonzero(((behind != 0) & ~self.solid).reshape(-1)).reshape(-1)
            if n.numel() == 0:
                self.links.append(None)
                continue
            xi, yi, zi = n % nx, (n // nx) % ny, n // (nx * ny)
            at = lambda k: ((xi + k * ei[0]) % nx) + nx * (
                ((yi + k * ei[1]) % ny) + ny * ((zi + k * ei[2]) % nz))
            inside = lambda k: self.in_domain(xi + k * ei[0], yi + k * ei[1], zi + k * ei[2])
            nff, nfff = at(1), at(2)
            flat_sid = sid.reshape(-1)
            ff = (flat_sid[nff] == 0) & inside(1)
            fff = ff & (flat_sid[nfff] == 0) & inside(2)
            who = behind.reshape(-1)[n].long() - 1
            q = torch.zeros(n.shape, dtype=torch.float64, device="cuda")
            arm = torch.zeros((3,) + tuple(n.shape), dtype=torch.float64, device="cuda")
            uw = torch.zeros_like(arm)
            for s, b in enumerate(self.p.solids):
                m = who == s
                flat = self.D == 2 or b.kind == W.CYLINDER_Z
                r = self.rel(s, xi[m].double(), yi[m].double(), zi[m].double())
                d = (-ei[0], -ei[1], 0 if flat else -ei[2])
                A = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
                if A > 0:
                    B = 2 * (r[0] * d[0] + r[1] * d[1] + r[2] * d[2])
                    Cc = r[0] ** 2 + r[1] ** 2 + r[2] ** 2 - b.radius ** 2
                    disc = torch.sqrt(torch.clamp(B * B - 4 * A * Cc, min=0))
                    qs = (-B + disc if b.fluid_inside else -B - disc) / (2 * A)
                else:
                    qs = torch.full_like(r[0], 0.5)
                qs = torch.clamp(qs, 1e-12, 1.0)
                q[m] = qs
                ar = [r[0] - qs * ei[0], r[1] - qs * ei[1], 0 * qs if flat else r[2] - qs * ei[2]]
                U, Om = self.U[s], self.Om[s]
                us = [U[0] + Om[1] * ar[2] - Om[2] * ar[1], U[1] + Om[2] * ar[0] - Om[0] * ar[2],
                      U[2] + Om[0] * ar[1] - Om[1] * ar[0]]
                for k in range(3):
                    arm[k][m] = ar[k]
                    uw[k][m] = us[k] if k < self.D else 0.0
            self.links.append((n, nff, nfff, ff, fff, q, arm, uw, who))

    def in_domain(self, x, y, z):
        ok = torch.ones_like(x, dtype=torch.bool)
        if self.p.faces is None:
            return ok
        for a, v in enumerate((x, y, z)):
            if self.p.faces[2 * a] != W.PERIODIC:
                ok &= (v >= 0) & (v < self.len[a])
        return ok

    # -- forces and collision
    def forces(self, f):
        """The body force of the collision of f, and IBM's force record."""
        g = [gi * self.g_on for gi in self.p.g]
        if not self.ibm:
            return g, None
        ut = [sum(e[c] * t for e, t in zip(self.e, f) if e[c]) + 0.5 * g[c]
              for c in range(self.D)]
        fld = [torch.zeros(self.shape, dtype=torch.float64, device="cuda") for _ in range(self.D)]
        rec = np.zeros((len(self.p.solids), 6))
        parts = []
        for s, b in enumerate(self.p.solids):
            RL = b.radius + self.p.retraction * (1 if b.fluid_inside else -1)
            dens = self.p.marker_density
            if self.D == 3 and b.kind == W.SPHERE:
                area = 4 * math.pi * RL * RL
                m = max(1, int(dens * area + 0.5))
                k = np.arange(m)
                zz = 1 - (2.0 * k + 1) / m
                rr = np.sqrt(1 - zz * zz)
                ga = math.pi * (3 - math.sqrt(5.0))
                dirs, dV = np.stack([rr * np.cos(ga * k), rr * np.sin(ga * k), zz]), area / m
            else:
                circ = 2 * math.pi * RL
                m = max(1, int(dens * circ + 0.5))
                th = 2 * math.pi * np.arange(m) / m
                dirs, dV = np.stack([np.cos(th), np.sin(th), 0 * th]), circ / m
            r = torch.from_numpy(RL * dirs).cuda()
            X = r + torch.tensor(self.c[s], dtype=torch.float64, device="cuda").view(3, 1)
            base = torch.floor(X) - 1
            idx, wgt = [], []
            for c in range(self.D):
                o = torch.arange(4, device="cuda").view(4, 1)
                d = (base[c] + o - X[c]).abs()
                near = (3 - 2 * d + torch.sqrt(torch.clamp(1 + 4 * d - 4 * d * d, min=0))) / 8
                far = (5 - 2 * d - torch.sqrt(torch.clamp(-7 + 12 * d - 4 * d * d, min=0))) / 8
                wgt.append(torch.where(d >= 2, 0 * d, torch.where(d >= 1, far, near)))
                idx.append((base[c].long() + o) % self.len[c])
            if self.D == 3:
                node = idx[0].view(1, 1, 4, m) + self.len[0] * (
                    idx[1].view(1, 4, 1, m) + self.len[1] * idx[2].view(4, 1, 1, m))
                wg = wgt[0].view(1, 1, 4, m) * wgt[1].view(1, 4, 1, m) * wgt[2].view(4, 1, 1, m)
            else:
                node = idx[0].view(1, 4, m) + self.len[0] * idx[1].view(4, 1, m)
                wg = wgt[0].view(1, 4, m) * wgt[1].view(4, 1, m)
            U, Om = self.U[s], self.Om[s]
            Ud = [U[0] + Om[1] * r[2] - Om[2] * r[1], U[1] + Om[2] * r[0] - Om[0] * r[2],
                  U[2] + Om[0] * r[1] - Om[1] * r[0]]
            parts.append((node.reshape(-1, m), wg.reshape(-1, m), dV, Ud, r,
                          [torch.zeros(m, dtype=torch.float64, device="cuda") for _ in range(3)]))
        for _ in range(max(1, self.p.ibm_iters)):
            new = []
            for node, wg, dV, Ud, r, Fm in parts:
                new.append([Ud[c] - (wg * (ut[c] + fld[c]).reshape(-1)[node]).sum(0)
                            for c in range(self.D)])
            for (node, wg, dV, Ud, r, Fm), dF in zip(parts, new):
                for c in range(self.D):
                    Fm[c] += dF[c]
                    fld[c].reshape(-1).index_add_(0, node.reshape(-1),
                                                  (dV * dF[c] * wg).reshape(-1))
        for s, (node, wg, dV, Ud, r, Fm) in enumerate(parts):
            Fs = [-dV * v for v in Fm]
            t = [r[1] * Fs[2] - r[2] * Fs[1], r[2] * Fs[0] - r[0] * Fs[2],
                 r[0] * Fs[1] - r[1] * Fs[0]]
            rec[s] = [float(v.sum()) for v in Fs + t]
        return [g[c] + fld[c] if c < self.D else g[c] for c in range(3)], rec

    def velocity(self, f, F):
        return [sum(e[c] * t for e, t in zip(self.e, f) if e[c]) + 0.5 * F[c]
                if c < self.D else torch.zeros_like(f[0]) for c in range(3)]

    def collide(self, f, F):
        """In place (the list's tensors are overwritten)."""
        om, cf = self.omega, 1.0 - 0.5 * self.omega
        drho = sum(f)
        u = self.velocity(f, F)
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        rows = []
        if self.mrt:
            for a in range(self.D):
                rows.append([((5 if self.D == 3 else 3) * sum(c * c for c in e) -
                              (9 if self.D == 3 else 5)) * e[a] for e in self.e])
        m = [torch.zeros_like(drho) for _ in rows]
        for i, (e, w) in enumerate(zip(self.e, self.w)):
            eu, eF = _edot(e, u), _edot(e, [v + 0 * drho for v in F])
            feq = w * (drho + 3 * eu + 4.5 * eu * eu - 1.5 * uu)
            fb = w * (3 * (eF - uF) + 9 * eu * eF)
            for a, row in enumerate(rows):
                if row[i]:
                    m[a] += row[i] * (f[i] - feq + 0.5 * fb)
            f[i] = f[i] - om * (f[i] - feq) + cf * fb
        for a, row in enumerate(rows):
            k = (om - self.sq) / sum(v * v for v in row)
            for i in range(self.Q):
                if row[i]:
                    f[i] += (k * row[i]) * m[a]
        return f

    # -- domain faces
    def faces(self, i, fi):
        """Replace the pulled f_i on links that leave the domain; returns the
        outflow region's rule, to be applied when every f_i is known."""
        p, ei = self.p, self.e[i]
        crossed = [(a, 2 * a if ei[a] > 0 else 2 * a + 1) for a in range(self.D)
                   if ei[a] and p.faces[2 * a] != W.PERIODIC]
        later = []
        for sub in range(1, 1 << len(crossed)):
            K = [crossed[k] for k in range(len(crossed)) if (sub >> k) & 1]
            rest = [crossed[k] for k in range(len(crossed)) if not (sub >> k) & 1]
            sl = [slice(None)] * 3  # z, y, x
            for a, k in K:
                sl[2 - a] = slice(0, 1) if k % 2 == 0 else slice(self.len[a] - 1, self.len[a])
            for a, k in rest:
                sl[2 - a] = slice(1, None) if k % 2 == 0 else slice(0, self.len[a] - 1)
            sl = tuple(sl)
            vel = [k for _, k in sorted(K, key=lambda t: t[1]) if p.faces[k] == W.VELOCITY]
            if vel:
                uf = p.u_face[vel[0]]
                fi[sl] = self.post[self.opp[i]][sl] + 6 * self.w[i] * sum(
                    ei[c] * uf[c] for c in range(self.D))
            elif any(p.faces[k] == W.CONVECTIVE for _, k in K):
                later.append(sl)
            else:
                axes = [a for a, _ in K]
                j = self.e.index(tuple(-ei[c] if c in axes else ei[c] for c in range(3)))
                plane = [slice(None)] * 3
                for a, k in K:
                    plane[2 - a] = sl[2 - a]
                t = self.post[j][tuple(plane)]
                t = torch.roll(t, tuple(ei[c] if c not in axes else 0 for c in (2, 1, 0)),
                               (0, 1, 2))
                cut = [slice(None)] * 3
                for a, k in rest:
                    cut[2 - a] = sl[2 - a]
                fi[sl] = t[tuple(cut)]
        return later

    def outlet(self):
        k = list(self.p.faces).index(W.CONVECTIVE)
        a, hi = k // 2, k % 2
        sl, inn = [slice(None)] * 3, [slice(None)] * 3
        n = self.len[a]
        sl[2 - a] = slice(n - 1, n) if hi else slice(0, 1)
        inn[2 - a] = slice(n - 2, n - 1) if hi else slice(1, 2)
        return a, (1.0 if hi else -1.0), tuple(sl), tuple(inn)

    def keep_outlet(self, f, F):
        a, sg, sl, _ = self.outlet()
        self.kept = [t[sl].clone() for t in f]
        j = sum(e[a] * t for e, t in zip(self.e, self.kept) if e[a])
        Fa = F[a]
        self.kept_u = sg * (j + 0.5 * (Fa[sl] if torch.is_tensor(Fa) else Fa))

    # -- one step
    def step(self):
        p = self.p
        if self.ibm and self.moving:
            self.advance()
        if self.moving:
            old = self.sid
            self.geometry()
            if not self.ibm:
                self.refill(old)
        flow_out = p.faces is not None and W.CONVECTIVE in p.faces
        f, later = [], []
        for i, ei in enumerate(self.e):
            fi = torch.roll(self.post[i], (ei[2], ei[1], ei[0]), (0, 1, 2))
            if p.faces is not None and i:
                later += [(i, sl) for sl in self.faces(i, fi)]
            f.append(fi)
        if flow_out:
            a, sg, sl0, inn = self.outlet()
            U = torch.clamp(self.kept_u, min=0)
            for i, sl in later:
                sel, isel = list(sl), list(sl)
                sel[2 - a], isel[2 - a] = slice(None), inn[2 - a]
                sel = tuple(sel)
                f[i][sl] = (self.kept[i][sel] + U[sel] * f[i][tuple(isel)]) / (1 + U[sel])
        rec = np.zeros((max(1, len(p.solids)), 6))
        flat = [t.reshape(-1) for t in self.post]
        vals = []
        for i in range(1, self.Q):
            if self.ibm or self.links[i - 1] is None:
                continue
            n, nff, nfff, ff, fff, q, arm, uw, who = self.links[i - 1]
            ei, ib, w = self.e[i], self.opp[i], self.w[i]
            mw = 6 * w * (ei[0] * uw[0] + ei[1] * uw[1] + ei[2] * uw[2])
            A, B = flat[ib], flat[i]
            if p.scheme == W.ZHAO_YONG:
                v = (2 * q * B[n] + self.pre[ib].reshape(-1)[n] + mw) / (1 + 2 * q)
            else:
                near = q < 0.5
                lin = torch.where(near, 2 * q * A[n] + (1 - 2 * q) * A[nff] + mw,
                                  (A[n] + mw) / (2 * q) + (2 * q - 1) / (2 * q) * B[n])
                v = torch.where(ff, lin, A[n] + mw)
                if p.scheme == W.BOUZIDI_QUAD:
                    k0 = 1 / (q * (2 * q + 1))
                    quad = torch.where(
                        near, q * (2 * q + 1) * A[n] + (1 + 2 * q) * (1 - 2 * q) * A[nff] -
                        q * (1 - 2 * q) * A[nfff] + mw,
                        k0 * (A[n] + mw) + (2 * q - 1) / q * B[n] +
                        (1 - 2 * q) / (2 * q + 1) * B[nff])
                    v = torch.where(ff & fff, quad, v)
            vals.append((i, n, v))
            full_out, full_in = A[n] + w, v + w
            dp = [full_out * (-ei[c] - uw[c]) - full_in * (ei[c] - uw[c]) for c in range(3)]
            tq = [arm[1] * dp[2] - arm[2] * dp[1], arm[2] * dp[0] - arm[0] * dp[2],
                  arm[0] * dp[1] - arm[1] * dp[0]]
            for s in range(len(p.solids)):
                m = (who == s).double()
                rec[s] += [float((v0 * m).sum()) for v0 in dp + tq]
        for i, n, v in vals:
            f[i].reshape(-1)[n] = v
        if self.pre is not None:
            self.pre = [t.clone() for t in f]
        F, ibm_rec = self.forces(f)
        self.force = rec if ibm_rec is None else ibm_rec
        if flow_out:
            self.keep_outlet(f, F)
        self.f_pre = None
        self.f = [t.clone() for t in f] if self.keep_f else None
        self.F = F
        new = self.collide(f, F)
        if bool(self.solid.any()):
            for i in range(self.Q):
                new[i] = torch.where(self.solid, self.other[i], new[i])
        self.other, self.post = self.post, new
        if self.moving and not self.ibm:
            self.advance()

    keep_f = False

    def advance(self):
        for s, b in enumerate(self.p.solids):
            if self.rho_p > 0:  # a free circle under bounce-back (Eq. 20)
                V = math.pi * b.radius ** 2
                mass = self.rho_p * V
                inertia = 0.5 * mass * b.radius ** 2
                for a in range(2):
                    new = self.U[s][a] + (self.force[s][a] +
                                          (self.rho_p - 1) * V * self.grav[a]) / mass
                    self.c[s][a] += 0.5 * (self.U[s][a] + new)
                    self.U[s][a] = new
                self.Om[s][2] += self.force[s][5] / inertia
            else:
                for a in range(3):
                    self.c[s][a] += self.U[s][a]

    def refill(self, old):
        """Uncovered nodes: the equilibrium at the mean density of the
        neighbours fluid before and after, at the wall velocity, collided."""
        fresh = torch.nonzero(((old != 0) & (self.sid == 0)).reshape(-1)).reshape(-1)
        if fresh.numel() == 0:
            return
        nx, ny, nz = self.len
        x, y, z = fresh % nx, (fresh // nx) % ny, fresh // (nx * ny)
        good = ((old == 0) & (self.sid == 0)).reshape(-1)
        flat = [t.reshape(-1) for t in self.post]
        tot = torch.zeros(fresh.shape, dtype=torch.float64, device="cuda")
        cnt = torch.zeros_like(tot)
        for e in self.e[1:]:
            nb = (x + e[0]) % nx + nx * ((y + e[1]) % ny + ny * ((z + e[2]) % nz))
            ok = good[nb].double()
            tot += ok * (1 + sum(t[nb] for t in flat))
            cnt += ok
        rho = torch.where(cnt > 0, tot / torch.clamp(cnt, min=1), torch.ones_like(tot))
        who = old.reshape(-1)[fresh].long() - 1
        u = [torch.zeros_like(tot) for _ in range(3)]
        for s in range(len(self.p.solids)):
            m = (who == s).double()
            r = self.rel(s, x.double(), y.double(), z.double())
            U, Om = self.U[s], self.Om[s]
            us = [U[0] + Om[1] * r[2] - Om[2] * r[1], U[1] + Om[2] * r[0] - Om[0] * r[2],
                  U[2] + Om[0] * r[1] - Om[1] * r[0]]
            for c in range(self.D):
                u[c] += m * us[c]
        new = self.collide(_feq(self.e, self.w, rho - 1, u), [0 * tot + g for g in self.p.g])
        for t, v in zip(flat, new):
            t[fresh] = v


def _stacked(r):
    scale = 1024.0 if r.p.precision == W.FP32_FP16 else 1.0
    return torch.stack([t.reshape(-1) * scale for t in r.post])


def _start(case, p, seed, k):
    if _starts_uniform(case):
        e, w = _lattice(p)
        z = torch.zeros(_shape(p), dtype=torch.float64, device="cuda")
        return _Ref(p, _feq(e, w, z, [z + v for v in p.u_face[0]]), True)
    return _Ref(p, _initial(p, seed, k), False)


def exact(case, seed):
    kind, n = case["kind"], case.get("steps", 0)
    ps = _problems(case, seed)
    outs = []
    for k, p in enumerate(ps):
        r = _start(case, p, seed, k)
        if kind == "settling":
            r.rho_p, r.grav, r.moving = 1.03, _gravity(case), True
        if kind in ("couette", "sphere", "moving", "open", "batch"):
            for _ in range(n):
                r.step()
            outs.append({"f": _stacked(r), "force": r.force[0][:3], "torque": r.force[0][3:]})
        elif kind == "steady":
            u0 = r.velocity(r.f, r.F)
            for j in range(n):
                r.keep_f = j == n - 1
                r.step()
            u1 = r.velocity(r.f, r.F)
            ns = (~r.solid).double()
            num = sum(((a - b) ** 2 * ns).sum() for a, b in zip(u1, u0))
            den = sum((a ** 2 * ns).sum() for a in u1)
            outs.append({"f": _stacked(r), "steps": n,
                         "residual": np.array([math.sqrt(float(num) / float(den))])})
        elif kind == "settling":
            for _ in range(n):
                r.step()
            outs.append({"f": _stacked(r), "centre": np.array(r.c[0]), "velocity": np.array(r.U[0]),
                         "omega": np.array(r.Om[0])})
        elif kind == "pair":
            rec = []
            for _ in range(n):
                r.step()
                rec.append(r.force[0])
            outs.append((_stacked(r), torch.from_numpy(np.array(rec))))
        else:
            for j in range(2):
                r.keep_f = j == 1
                r.step()
            outs.append(_fields(r))
    if kind == "batch":
        return {"lattice%02d" % k: o for k, o in enumerate(outs)}
    if kind == "pair":
        return {"f_ibb": outs[0][0], "f_ibm": outs[1][0], "record_ibb": outs[0][1],
                "record_ibm": outs[1][1]}
    return outs[0]


def _fields(r):
    """Velocity, strain rate (xx yy zz xy yz xz) and dissipation rate."""
    F = [v + torch.zeros_like(r.f[0]) for v in r.F]
    u = r.velocity(r.f, F)
    feq = _feq(r.e, r.w, sum(r.f), u)
    P = {}
    for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2)):
        P[a, b] = 0.5 * (F[a] * u[b] + u[a] * F[b]) + sum(
            e[a] * e[b] * (f - q) for e, f, q in zip(r.e, r.f, feq) if e[a] * e[b])
    iso = (P[0, 0] + P[1, 1] + P[2, 2]) / 3
    ns = (~r.solid).double()
    S, ss = [], 0
    for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2)):
        # one rate for the stress and the trace: -1.5 omega P
        s = -1.5 * r.omega * ((P[a, b] - iso if a == b else P[a, b]) + (iso if a == b else 0.0))
        S.append((s * ns).reshape(-1))
        ss = ss + (1 if a == b else 2) * s * s
    nu = (r.p.tau - 0.5) / 3
    return {"velocity": torch.stack([(v * ns).reshape(-1) for v in u]).view(3, *r.shape).reshape(3, -1),
            "strain": torch.stack(S), "dissipation": (2 * nu * ss * ns).reshape(1, -1)}
