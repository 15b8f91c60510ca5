"""What the speed of this framework is judged by: whole runs of the solver
through its public entry points (`Grid`, `Batch` and, for device-resident
fields of a batch, the C ABI), and the same runs in plain 64-bit torch.

One pass is what a user's program does with one problem: give the grid its
primitive fields (device-resident FP64 planes), set the body where it moves,
run a number of steps with the time step computed on the device, and read the
result: the conserved state in place (`state_layout`) or, for a batch, copied
out.  Steps are few, so that a pass stays short; the flow is developed, not
two constant states: every field carries smooth disturbances (sound waves and
density waves of about 1 %), so that every cell and face has work to do.

    tube     1-D shock running at a rigid wall; the smallest calls
    cylinder 2-D shock over a rigid cylinder in air
    wedge    2-D strong shock up a rigid wedge standing on a reflective floor
    batch    2-D many independent shock-over-ellipse problems of mixed sizes
    pool     2-D free body in shocked air over water (two materials; drawn
             cases also three), driven by the pressure force
    impact   2-D elastoplastic block striking a rigid wedge; aluminium, or
             copper with Johnson-Cook flow stress and plastic-strain planes
    sphere   3-D shock over a rigid sphere

Outputs are grouped as the reduced system groups its variables: volume
fractions, partial densities, momenta, energy, stretch tensor, rigid field,
plastic strains, and the simulated time (and the body's state where it moves).
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2111_11806_gb300 import binding as B

AIR = dict(kind="ideal", gamma=1.4, rho0=1.225)
GAS = dict(kind="ideal", gamma=1.4)
WATER = dict(kind="stiffened", gamma=4.4, pinf=6.0e8, rho0=1000.0)
HELIUM = dict(kind="ideal", gamma=1.67, rho0=0.166)
ALUMINIUM = dict(kind="romenskii", rho0=2700.0, K0=76.0e9, G0=26.0e9, alpha=0.627, beta=2.288, Gamma0=1.484,
                 sigY=0.3e9)
COPPER = dict(kind="romenskii", rho0=8960.0, K0=130.1e9, G0=43.33e9, alpha=1.0, beta=3.0, Gamma0=2.0,
              jc_c1=0.09e9, jc_c2=0.292e9, jc_c3=0.025, jc_n=0.31, jc_m=1.09, jc_tmelt=1358.0, jc_cv=385.0)
PURE = 1.0e-8      # residual volume fraction of an absent material
BATCH_SIZES = (128, 192, 256, 384, 512)


def listed():
    return [
        # a 1-D study: the smallest grid of the tests, default precision; all launch latency
        dict(name="tube_400_fp64", flow="tube", n0=400, fp32=False, steps=60),
        # the benchmark's single 2-D grid, in both precisions; FP64 (the default) at an odd size
        dict(name="cylinder_512_fp32", flow="cylinder", n0=512, n1=512, fp32=True, steps=30),
        dict(name="cylinder_383x401_fp64", flow="cylinder", n0=383, n1=401, fp32=False, steps=6),
        # the paper's wedge test at its finest level: reflective floor, rows that are no multiple of a strip
        dict(name="wedge_1200x800_fp32", flow="wedge", n0=1200, n1=800, fp32=True, steps=20),
        # the headline: 256 independent problems of 128^2 to 512^2, 26 million cells
        dict(name="batch_256_fp32", flow="batch", count=256, fp32=True, steps=16),
        # a smaller design study in FP64
        dict(name="batch_16_fp64", flow="batch", count=16, fp32=False, steps=3),
        # the benchmark's dynamic body, two fluids, in both precisions
        dict(name="pool_1024x512_fp32", flow="pool", n0=1024, n1=512, nmat=2, fp32=True, steps=6),
        dict(name="pool_501x250_fp64", flow="pool", n0=501, n1=250, nmat=2, fp32=False, steps=4),
        # the benchmark's elastoplastic impact
        dict(name="impact_1024_fp32", flow="impact", n0=1024, n1=1024, copper=False, fp32=True, steps=6),
        # copper with hardening, softening and plastic-strain planes, FP64
        dict(name="copper_301x299_fp64", flow="impact", n0=301, n1=299, copper=True, fp32=False, steps=2),
        # the benchmark's 3-D grid; FP64 at a ragged size
        dict(name="sphere_256_fp32", flow="sphere", n0=256, n1=256, n2=256, fp32=True, steps=5),
        dict(name="sphere_97x90x101_fp64", flow="sphere", n0=97, n1=90, n2=101, fp32=False, steps=2),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: a flow, a precision, sizes spread over their logarithm,
    and the options a flow is used with (periodic or walled sides, a moving
    body, three materials, MUSCL only)."""
    flow = rng.choice(("tube", "cylinder", "cylinder", "wedge", "batch", "pool", "pool", "impact", "sphere", "sphere"))
    fp32 = rng.random() < 0.5
    if flow == "tube":
        return dict(flow=flow, n0=_between(rng, 100, 20000), fp32=fp32, steps=rng.randint(20, 80))
    if flow == "cylinder":
        c = dict(flow=flow, n0=_between(rng, 64, 1600 if fp32 else 500), n1=_between(rng, 64, 1600 if fp32 else 500),
                 fp32=fp32, steps=rng.randint(4, 20) if fp32 else rng.randint(2, 6))
        kind = rng.choice(("plain", "plain", "moving", "periodic"))
        if kind != "plain":
            c[kind] = True
        return c
    if flow == "wedge":
        n0 = _between(rng, 150, 1500 if fp32 else 480)
        return dict(flow=flow, n0=n0, n1=n0 * 2 // 3, fp32=fp32, steps=rng.randint(4, 20) if fp32 else rng.randint(2, 5))
    if flow == "batch":
        return dict(flow=flow, count=_between(rng, 2, 128 if fp32 else 16), fp32=fp32, steps=rng.randint(4, 16) if fp32
                    else rng.randint(1, 3))
    if flow == "pool":
        n0 = _between(rng, 128, 1400 if fp32 else 480)
        return dict(flow=flow, n0=n0, n1=max(60, int(n0 * rng.uniform(0.4, 0.7))), nmat=rng.choice((2, 2, 3)), fp32=fp32,
                    steps=rng.randint(3, 8) if fp32 else rng.randint(1, 4), thinc=rng.random() < 0.8)
    if flow == "impact":
        n0 = _between(rng, 120, 1100 if fp32 else 300)
        return dict(flow=flow, n0=n0, n1=max(100, int(n0 * rng.uniform(0.7, 1.2))), copper=rng.random() < 0.4, fp32=fp32,
                    steps=rng.randint(2, 5) if fp32 else rng.randint(1, 2))
    n = [_between(rng, 40, 200 if fp32 else 90) for _ in range(3)]
    c = dict(flow=flow, n0=n[0], n1=n[1], n2=n[2], fp32=fp32, steps=rng.randint(2, 5) if fp32 else 2)
    if rng.random() < 0.3:
        c["moving"] = True
    return c


# ------------------------------------------------------------------ problems

def _layout(dim, nmat, solid, history):
    nv = (3 if dim == 1 else 5 if dim == 2 else 9) if solid else 0
    iu = 2 * nmat - 1
    ir = iu + dim + 1 + nv
    return dict(phi=(0, nmat - 1), mass=(nmat - 1, nmat), momentum=(iu, dim), energy=(iu + dim, 1),
                stretch=(iu + dim + 1, nv), rigid=(ir, 1), strain=(ir + 1, nmat if history else 0),
                nvar=ir + 1 + (nmat if history else 0))


def _shock(mach, gamma, rho, p):
    """Density, velocity and pressure behind a shock of Mach number `mach`."""
    p2 = p * (1 + 2 * gamma / (gamma + 1) * (mach * mach - 1))
    r2 = rho * (gamma + 1) * mach * mach / ((gamma - 1) * mach * mach + 2)
    return r2, mach * math.sqrt(gamma * p / rho) * (1 - rho / r2), p2


class _Problem:
    """Grid, materials, body and FP64 primitive planes of one problem; the
    planes are made on `dev` from the numbers that `rng` gives."""

    def __init__(self, case, rng, dev, n=None):
        self.case = case
        f = case["flow"]
        self.dim = dim = 1 if f == "tube" else 3 if f == "sphere" else 2
        self.n = n or tuple(case["n%d" % d] for d in range(dim))
        self.solid = f == "impact"
        self.history = self.solid and case["copper"]
        self.periodic, self.walls = [0] * dim, [0] * 6
        self.lo, self.hi = [0.0] * dim, [1.0] * dim
        self.cfl, self.v, self.x, self.mass, self.dynamic = 0.8, (0.0, 0.0, 0.0), (0.0, 0.0, 0.0), 0.0, False
        self.mats = [AIR]
        if f == "wedge":
            self.mats, self.hi, self.walls, self.cfl = [GAS], [3.0, 2.0], [0, 0, 1, 0, 0, 0], 0.4
        if f == "pool":
            self.mats = [WATER, AIR] if case["nmat"] == 2 else [WATER, HELIUM, AIR]
            self.hi = [2.0, 1.0]
        if f == "impact":
            self.mats = [COPPER if case["copper"] else ALUMINIUM, AIR]
            self.hi = [0.1, 0.1]
        if case.get("periodic"):
            self.periodic[1] = 1
        self.dx = [(self.hi[d] - self.lo[d]) / self.n[d] for d in range(dim)]
        self.lay = _layout(dim, len(self.mats), self.solid, self.history)
        getattr(self, "_" + f)(case, rng, dev)

    def _waves(self, rng, amp, X):
        """1 + amp * (three smooth waves), of wavelengths of 1/2 to 1/6 of the domain."""
        s = torch.zeros_like(X[0])
        for _ in range(3):
            a = sum(2 * math.pi * rng.integers(1, 6) / (self.hi[d] - self.lo[d]) * X[d] for d in range(self.dim))
            s = s + torch.sin(a + rng.uniform(0, 2 * math.pi))
        return 1 + amp / 3 * s

    def _centres(self, dev):
        ax = [self.lo[d] + (torch.arange(self.n[d], dtype=torch.float64, device=dev) + 0.5) * self.dx[d]
              for d in range(self.dim)]
        return [m.reshape(-1) for m in torch.meshgrid(*ax[::-1], indexing="ij")][::-1]    # x fastest

    def _gas(self, rng, dev, X, mach, x_shock, rho, p, back=False):
        """Gas shocked left of x_shock and moving right (right of it and moving
        left with `back`), disturbed; returns the planes."""
        w = torch.zeros(self.lay["nvar"], X[0].numel(), dtype=torch.float64, device=dev)
        g = self.mats[-1]["gamma"]
        r2, u2, p2 = _shock(mach, g, rho, p)
        post = X[0] > x_shock if back else X[0] < x_shock
        u2 = -u2 if back else u2
        c = math.sqrt(g * p / rho)
        w[self.lay["mass"][0] + len(self.mats) - 1] = torch.where(post, r2, rho) * self._waves(rng, 0.02, X)
        iu = self.lay["momentum"][0]
        for d in range(self.dim):
            w[iu + d] = 0.02 * c * (self._waves(rng, 1.0, X) - 1)
        w[iu] += torch.where(post, u2, 0.0)
        w[self.lay["energy"][0]] = torch.where(post, p2, p) * self._waves(rng, 0.02, X)
        return w

    def _rigid(self, dist):
        return 0.5 * (1 - torch.tanh(dist / min(self.dx)))

    def _tube(self, case, rng, dev):
        X = self._centres(dev)
        w = self._gas(rng, dev, X, rng.uniform(1.8, 2.2), 0.6, 1.225, 1.0e5)
        w[self.lay["rigid"][0]] = self._rigid(rng.uniform(0.66, 0.7) - X[0])
        self.prim = w

    def _cylinder(self, case, rng, dev):
        X = self._centres(dev)
        w = self._gas(rng, dev, X, rng.uniform(2.5, 3.0), 0.36, 1.225, 1.0e5)
        at = (rng.uniform(0.48, 0.52), rng.uniform(0.48, 0.52))
        w[self.lay["rigid"][0]] = self._rigid(torch.hypot(X[0] - at[0], X[1] - at[1]) - 0.1)
        if case.get("moving"):
            self.v = (rng.uniform(-60, -20), rng.uniform(10, 40), 0.0)
        self.prim = w

    def _wedge(self, case, rng, dev):
        X = self._centres(dev)
        w = self._gas(rng, dev, X, rng.uniform(9.0, 10.0), 0.6, 1.4, 1.0)
        th = math.radians(rng.uniform(27, 33))
        sx, sy = X[0] - 0.5, X[1]
        along, above = sx * math.cos(th) + sy * math.sin(th), -sx * math.sin(th) + sy * math.cos(th)
        w[self.lay["rigid"][0]] = self._rigid(torch.where(along >= 0, above, torch.hypot(sx, sy)))
        self.prim = w

    def _batch(self, case, rng, dev):
        X = self._centres(dev)
        w = self._gas(rng, dev, X, rng.uniform(1.5, 3.0), 0.34, 1.225, 1.0e5)
        a, b, th = rng.uniform(0.05, 0.15), rng.uniform(0.05, 0.15), rng.uniform(0, math.pi)
        xr = (X[0] - 0.5) * math.cos(th) + (X[1] - 0.5) * math.sin(th)
        yr = -(X[0] - 0.5) * math.sin(th) + (X[1] - 0.5) * math.cos(th)
        F = torch.sqrt((xr / a) ** 2 + (yr / b) ** 2).clamp_min(1e-30)
        grad = torch.hypot(xr / (a * a * F), yr / (b * b * F)).clamp_min(1e-30)
        w[self.lay["rigid"][0]] = self._rigid((F - 1) / grad)
        self.prim = w

    def _pool(self, case, rng, dev):
        X = self._centres(dev)
        w = self._gas(rng, dev, X, rng.uniform(2.8, 3.0), 0.5, 1.225, 1.0e5, back=True)
        N, r = len(self.mats), self.lay["mass"][0]
        iu, ir = self.lay["momentum"][0], self.lay["rigid"][0]
        water = X[1] < 0.03
        bubble = torch.hypot(X[0] - 1.2, X[1] - 0.4) < 0.15
        w[0] = torch.where(water, 1 - (N - 1) * PURE, PURE)
        w[r] = 1000.0 * self._waves(rng, 1e-4, X)
        if N == 3:
            w[1] = torch.where(bubble & ~water, 1 - (N - 1) * PURE, PURE)
            w[r + 1] = 0.166 * self._waves(rng, 0.02, X)
        # the shock runs at the body, at rest in the air over the water; faint waves in the water
        w[iu] = torch.where(water | (X[0] < 0.5), 0.2 * (self._waves(rng, 1.0, X) - 1), w[iu])
        w[iu + 1] = 0.2 * (self._waves(rng, 1.0, X) - 1)
        self.x = (rng.uniform(0.14, 0.16), rng.uniform(0.05, 0.06), 0.0)
        w[ir] = self._rigid(torch.hypot(X[0] - self.x[0], X[1] - self.x[1]) - 0.05)
        self.mass, self.dynamic = 7.6 * 1.225 * math.pi * 0.05 ** 2, True
        self.prim = w

    def _impact(self, case, rng, dev):
        X = self._centres(dev)
        w = self._gas(rng, dev, X, 1.0, -1.0, 1.225, 1.0e5)
        iu, ip, iv = self.lay["momentum"][0], self.lay["energy"][0], self.lay["stretch"][0]
        tip = rng.uniform(0.058, 0.062)
        block = (X[0] >= tip - 0.035) & (X[0] <= tip - 0.004) & (X[1] >= 0.03) & (X[1] <= 0.07)
        w[0] = torch.where(block, 1 - PURE, PURE)
        w[self.lay["mass"][0]] = self.mats[0]["rho0"]
        # sheared and compressed by sound and shear waves within and beyond the elastic limit
        speed = rng.uniform(380, 420)
        w[iu] = torch.where(block, speed * self._waves(rng, 0.03, X), w[iu])
        w[iu + 1] = torch.where(block, 0.03 * speed * (self._waves(rng, 1.0, X) - 1), w[iu + 1])
        for k, (mean, amp) in enumerate(((1, 2e-3), (0, 2e-3), (0, 2e-3), (1, 2e-3), (1, 2e-3))):
            w[iv + k] = mean + amp * (self._waves(rng, 1.0, X) - 1)
        w[ip] = torch.where(block, 1.0e8 * self._waves(rng, 0.2, X), w[ip])
        th = math.radians(30)
        xi, eta = X[0] - tip, (X[1] - 0.05).abs()
        proj, line = xi * math.cos(th) + eta * math.sin(th), -xi * math.sin(th) + eta * math.cos(th)
        w[self.lay["rigid"][0]] = self._rigid(torch.where(proj >= 0, line, torch.hypot(xi, eta)))
        if self.history:
            w[self.lay["strain"][0]] = 0.02 * self._waves(rng, 0.5, X)
        self.prim = w

    def _sphere(self, case, rng, dev):
        X = self._centres(dev)
        w = self._gas(rng, dev, X, rng.uniform(2.2, 2.6), 0.36, 1.225, 1.0e5)
        at = [rng.uniform(0.48, 0.52) for _ in range(3)]
        w[self.lay["rigid"][0]] = self._rigid(sum((X[d] - at[d]) ** 2 for d in range(3)).sqrt() - 0.1)
        if case.get("moving"):
            self.v = (rng.uniform(-60, -20), rng.uniform(10, 40), rng.uniform(5, 30))
        self.prim = w

    @property
    def moves(self):
        return self.dynamic or any(self.v)


def _problems(case, seed, dev):
    rng = np.random.default_rng([2111, seed])
    if case["flow"] != "batch":
        return [_Problem(case, rng, dev)]
    # the instances' sizes belong to the case (they stay as inputs change), their flows to the seed
    sizes = np.random.default_rng(11806).choice(BATCH_SIZES, case["count"])
    return [_Problem(case, rng, dev, (int(n), int(n))) for n in sizes]


# ---------------------------------------------------------------------- passes

_the_stream = []


def _stream():
    """The one stream that the program runs its grids on (a step is a CUDA graph there)."""
    if not _the_stream:
        _the_stream.append(torch.cuda.Stream())
    return _the_stream[0]


class _Instance:
    """What `Batch` wants of a problem."""

    def __init__(self, p):
        self.dim, self.solid, self.materials, self.n = 2, False, p.mats, p.n
        self.lo, self.hi, self.periodic, self.walls, self.body_v = p.lo, p.hi, p.periodic, p.walls, p.v


def _groups(p, planes):
    """The planes of one state by kind of variable, each as (planes, nz, ny, nx)."""
    shape = tuple(p.n[::-1])
    out = {}
    for k in ("phi", "mass", "momentum", "energy", "stretch", "rigid", "strain"):
        at, count = p.lay[k]
        if count:
            out[k] = planes[at:at + count].reshape((count,) + shape)
    return out


def _body(case, p, force, v, x):
    """The free body's force, velocity and position.  In an FP32 run the position alone: in the few steps from rest
    the body gains centimetres per second, which the FP32 pressure of water (steps of 200 Pa) does not resolve."""
    if case["fp32"]:
        return dict(x=x[:p.dim].astype(np.float32))
    return dict(force=force[:p.dim], v=v[:p.dim], x=x[:p.dim])


def prepare(case, seed):
    dev = torch.device("cuda:0")
    ps = _problems(case, seed, dev)
    prec = B.DFV_FP32 if case["fp32"] else B.DFV_FP64
    torch.cuda.synchronize()
    if case["flow"] == "batch":
        b = B.Batch([_Instance(p) for p in ps], precision=prec, stream=_stream())
        nvar, cells = b.nvar, b.cells
        out = torch.empty(nvar * b.total_cells, dtype=torch.float64, device=dev)
        res = torch.empty_like(out, dtype=torch.float32) if case["fp32"] else out
        ends = np.cumsum([0] + [nvar * c for c in cells])
        ptr = ctypes.c_void_p * b.count
        s = dict(case=case, batch=b, prims=[p.prim for p in ps], out=out, res=res,
                 src=ptr(*[p.prim.data_ptr() for p in ps]), dst=ptr(*[out[int(e):].data_ptr() for e in ends[:-1]]),
                 parts=[res[int(a):int(e)].view(nvar, c) for a, e, c in zip(ends[:-1], ends[1:], cells)])
        assert B.load().dfv_batch_set_all_fields(b._h, s["src"], 1) == B.DFV_OK
        b.autotune(trial_steps=2, cfl=0.8)
        torch.cuda.synchronize()
        return s
    p = ps[0]
    g = B.Grid(p.dim, p.n, p.lo, p.hi, p.mats, solid=2 if p.history else p.solid, precision=prec, periodic=p.periodic,
               walls=p.walls, use_thinc=case.get("thinc", True), stream=_stream())
    g.set_body(p.v, p.x, p.mass, p.dynamic)
    off, pitch, nvar, size = g.state_layout()
    at = g.aligned_offset() + off[0]
    planes = g.workspace[at:at + nvar * pitch * size].view(torch.float32 if size == 4 else torch.float64)
    torch.cuda.synchronize()
    return dict(case=case, grid=g, problem=p, state=planes.view(nvar, pitch)[:, :g.ncell])


def run(state):
    case = state["case"]
    if "batch" in state:
        # the fields of every instance from and to device memory (the C call: the Python one takes host arrays);
        # an FP32 batch's result is kept in the FP32 values that it consists of
        b, lib = state["batch"], B.load()
        lib.dfv_batch_set_all_fields(b._h, state["src"], 1)
        b.run(case["steps"], 0.8)
        lib.dfv_batch_get_all_fields(b._h, state["dst"], B.DFV_FIELDS_CONSERVED, 1)
        if state["res"] is not state["out"]:
            with torch.cuda.stream(b.stream):
                state["res"].copy_(state["out"])
        return state["res"]
    g, p = state["grid"], state["problem"]
    g.set_fields(p.prim)
    if p.moves:
        g.set_body(p.v, p.x, p.mass, p.dynamic)
    t = g.run(case["steps"], p.cfl)
    out = _groups(p, state["state"])
    out["time"] = t
    if p.dynamic:
        out.update(_body(case, p, *g.body()))
    return out


def work(case):
    """Bytes: the given FP64 planes read once and the result written once, and
    a state that is larger than the cache (129 MB) read and written once a
    step.  Flops: additions, multiplications, divisions and roots of the
    scheme for each cell, stage and face, every slope, closure and flux
    computed once (about; a logarithm or power as 20)."""
    dim = 1 if case["flow"] == "tube" else 3 if case["flow"] == "sphere" else 2
    nmat = case.get("nmat", 2 if case["flow"] == "impact" else 1)
    solid = case["flow"] == "impact"
    lay = _layout(dim, nmat, solid, solid and case["copper"])
    nvar, w = lay["nvar"], 4 if case["fp32"] else 8
    if case["flow"] == "batch":
        cells = int(sum(int(n) ** 2 for n in np.random.default_rng(11806).choice(BATCH_SIZES, case["count"])))
    else:
        cells = math.prod(case["n%d" % d] for d in range(dim))
    closure = 10 * nmat + 4 * dim + (200 if solid else 0)
    face = 2 * closure + 30 + 8 * nvar + (40 if solid else 0)
    stage = closure + dim * (face + 8 * nvar) + 8 * nvar
    extra = 2 * closure + (150 if solid else 0)      # wave speeds; plastic return
    turns = case["steps"] if w * nvar * cells > 129e6 else 0
    return dict(bytes=cells * nvar * (8.0 + w + 2.0 * w * turns),
                flops=float(cells) * case["steps"] * (3 * stage + extra))


# ------------------------------------------------------- the scheme in 64 bits

class _Exact:
    """The scheme in plain torch FP64, for `b` problems of one size at a time:
    a state is a list of planes of shape (b, nz, ny, nx)."""

    def __init__(self, ps, use_thinc):
        p = ps[0]
        self.p, self.dim, self.N, self.thinc_on = p, p.dim, len(p.mats), use_thinc
        self.n = tuple(p.n) + (1,) * (3 - p.dim)
        self.dx, self.lay, self.nvar = p.dx, p.lay, p.lay["nvar"]
        self.b = len(ps)
        self.dev = p.prim.device
        self.iphi, self.iar, self.iu = 0, p.lay["mass"][0], p.lay["momentum"][0]
        self.iE, self.iv, self.nv, self.ir, self.ih = (p.lay["energy"][0], p.lay["stretch"][0], p.lay["stretch"][1],
                                                       p.lay["rigid"][0], p.lay["strain"][0])
        self.vmap = ((0, 0), (0, 1), (1, 0), (1, 1), (2, 2)) if self.nv else ()
        shape = (self.b, self.n[2], self.n[1], self.n[0])
        prim = torch.stack([q.prim for q in ps], 1)
        self.U = self.to_cons([prim[v].reshape(shape) for v in range(self.nvar)])
        self.v, self.x = list(p.v), list(p.x)
        self.force = [0.0] * 3
        self.t = 0.0

    # ---- closures
    def ref(self, m, rho, J2):
        """Gamma, e_ref, p_ref, de_ref/drho, dp_ref/drho, G of a material."""
        if m["kind"] != "romenskii":
            z = torch.zeros_like(rho)
            return m["gamma"] - 1, z, z - (m["gamma"] * m["pinf"] if m["kind"] == "stiffened" else 0.0), z, z, z
        al, be, K0, r0 = m["alpha"], m["beta"], m["K0"], m["rho0"]
        x = rho / r0
        xa = x ** al
        G = m["G0"] * x ** (be + 1)
        pr = -K0 / (2 * al * al) * (xa - 1) ** 2 + K0 / al * (xa - 1) * xa + be * G * J2
        dp = K0 / r0 * x ** (al - 1) * (2 * xa - 1 - (xa - 1) / al) + be * (be + 1) * G * J2 / rho
        return m["Gamma0"], K0 / (2 * rho * al * al) * (xa - 1) ** 2 + G * J2 / rho, pr, pr / rho ** 2, dp, G

    def hencky(self, A):
        """dev H (in-plane entries), J^2, the log-stretches and cos, sin of the
        doubled angle of their directions, of the planes xx, xy, yx, yy, zz."""
        b00, b01, b11 = A[0] ** 2 + A[1] ** 2, A[0] * A[2] + A[1] * A[3], A[2] ** 2 + A[3] ** 2
        mid, half = 0.5 * (b00 + b11), 0.5 * (b00 - b11)
        rad = torch.sqrt(half ** 2 + b01 ** 2)
        h = [0.5 * torch.log(mid + rad), 0.5 * torch.log(mid - rad), 0.5 * torch.log(A[4] ** 2)]
        hm = (h[0] + h[1] + h[2]) / 3
        d = [a - hm for a in h]
        one = torch.where(rad > 0, rad, torch.ones_like(rad))
        c2, s2 = torch.where(rad > 0, half / one, torch.ones_like(rad)), torch.where(rad > 0, b01 / one, torch.zeros_like(rad))
        av, df = 0.5 * (d[0] + d[1]), 0.5 * (d[0] - d[1])
        H = {(0, 0): av + df * c2, (1, 1): av - df * c2, (0, 1): df * s2, (1, 0): df * s2}
        return H, d[0] ** 2 + d[1] ** 2 + d[2] ** 2, d, c2, s2

    def fractions(self, w):
        phi = [w[self.iphi + l] for l in range(self.N - 1)]
        return phi + [1 - sum(phi)] if phi else [torch.ones_like(w[0])]

    def state(self, w):
        """Everything a face or a cell needs, from primitives."""
        s = dict(phi=[f.clamp(0, 1) for f in self.fractions(w)])
        rl = [w[self.iar + l] for l in range(self.N)]
        s["rl"], s["ar"] = rl, [f * r for f, r in zip(s["phi"], rl)]
        s["rho"] = sum(s["ar"])
        s["u"], s["p"] = [w[self.iu + a] for a in range(self.dim)], w[self.iE]
        s["eps"] = [w[self.ih + l] for l in range(self.N)] if self.p.history else None
        s["H"], J2 = None, torch.zeros_like(s["p"])
        if self.nv:
            s["H"], J2, s["d"], s["c2a"], s["s2a"] = self.hencky(w[self.iv:self.iv + self.nv])
        s["J2"] = J2
        rhoe = den = Gn = Sn = Yn = 0.0
        for l, m in enumerate(self.p.mats):
            Gam, e, pr, de, dp, G = self.ref(m, rl[l], J2)
            rhoe = rhoe + torch.where(s["ar"][l] != 0, s["ar"][l] * e, 0.0) + s["phi"][l] * (s["p"] - pr) / Gam
            den = den + s["phi"][l] / Gam
            Gn, Sn = Gn + s["phi"][l] * G / Gam, Sn + s["phi"][l] * m.get("sigY", 0.0) / Gam
            c2 = (Gam * s["p"] + s["p"] - pr) / rl[l] + dp - Gam * rl[l] * de + 4.0 / 3 * G / rl[l]
            Yn = Yn + torch.where(s["ar"][l] != 0, s["ar"][l] / s["rho"] * c2 / Gam, 0.0)
        s["rhoE"] = rhoe + 0.5 * s["rho"] * sum(u * u for u in s["u"])
        s["G"], s["sigY"], s["c"] = Gn / den, Sn / den, torch.sqrt(Yn / den)
        return s

    def to_cons(self, w):
        s = self.state(w)
        q = s["phi"][:self.N - 1] + s["ar"] + [s["rho"] * u for u in s["u"]] + [s["rhoE"]] + list(w[self.iv:self.ir + 1])
        return q + ([a * e for a, e in zip(s["ar"], s["eps"])] if self.p.history else [])

    def to_prim(self, q):
        phi, ar = self.fractions(q), [q[self.iar + l] for l in range(self.N)]
        rho = sum(ar)
        u = [q[self.iu + a] / rho for a in range(self.dim)]
        J2 = self.hencky(q[self.iv:self.iv + self.nv])[1] if self.nv else torch.zeros_like(rho)
        num, den, rl = q[self.iE] - 0.5 * rho * sum(a * a for a in u), 0.0, []
        for l, m in enumerate(self.p.mats):
            f = phi[l].clamp(0, 1)
            r = rho if self.N == 1 else ar[l] / f.clamp_min(1e-14)
            if self.N > 1 and m.get("rho0", 0.0) > 0:
                r = torch.where(f < 1e-6, m["rho0"], r)
            rl.append(r)
            Gam, e, pr, _, _, _ = self.ref(m, r, J2)
            num = num - torch.where(ar[l] != 0, ar[l] * e, 0.0) + f * pr / Gam
            den = den + f / Gam
        w = phi[:self.N - 1] + rl + u + [num / den] + list(q[self.iv:self.ir + 1])
        if self.p.history:
            w += [torch.where(a != 0, q[self.ih + l] / torch.where(a != 0, a, 1.0), 0.0) for l, a in enumerate(ar)]
        return w

    # ---- space
    def line(self, d, k):
        """Cells -k .. n+k-1 of direction d: their cells in the grid, and which are mirror images."""
        n, i = self.n[d], torch.arange(-k, self.n[d] + k, device=self.dev)
        flip = torch.zeros(i.shape, dtype=torch.bool, device=self.dev)
        if self.p.periodic[d]:
            return i % n, flip
        j = i.clamp(0, n - 1)
        for side, out in ((0, i < 0), (1, i > n - 1)):
            if self.p.walls[2 * d + side]:
                j = torch.where(out, (-1 - i if side == 0 else 2 * n - 1 - i).clamp(0, n - 1), j)
                flip = flip | out
        return j, flip

    @staticmethod
    def slope(m, c, p):
        a, b = c - m, p - c
        ab = a * b
        return torch.where(ab > 0, 2 * ab / torch.where(ab > 0, a + b, 1.0), 0.0)

    def thinc(self, qm, q0, qp, lo, hi):
        beta = 1.6
        mono = (qp - q0) * (q0 - qm) > 0
        qmin, dq = torch.minimum(qm, qp), (qp - qm).abs()
        th = torch.where(qp >= qm, 1.0, -1.0).to(torch.float64)
        C = (q0 - qmin) / torch.where(mono, dq, 1.0)
        ok = mono & (C > 1e-8) & (C < 1 - 1e-8)
        ty = (math.cosh(beta) - torch.exp(th * beta * (2 * C - 1))) / math.sinh(beta)
        tb = math.tanh(beta)
        t1 = (tb - ty) / (1 - tb * ty)
        return torch.where(ok, qmin + 0.5 * dq * (1 - th * ty), lo), torch.where(ok, qmin + 0.5 * dq * (1 + th * t1), hi)

    def faces(self, d, w):
        """Left and right primitives at the n+1 faces of direction d."""
        ax = 3 - d
        j, flip = self.line(d, 3)
        sgn = torch.where(flip, -1.0, 1.0).to(torch.float64).reshape([-1 if a == ax else 1 for a in range(4)])
        n = self.n[d]
        at = lambda q, k, c: q.narrow(ax, k, c)  # noqa: E731
        L, R = [], []
        for v in range(self.nvar):
            q = w[v].index_select(ax, j)
            odd = v == self.iu + d
            if self.iv <= v < self.iv + self.nv:
                a, b = self.vmap[v - self.iv]
                odd = (a == d) != (b == d)
            if odd:
                q = q * sgn
            qm, q0, qp = at(q, 0, n + 4), at(q, 1, n + 4), at(q, 2, n + 4)      # cells -2 .. n+1
            s = self.slope(qm, q0, qp)
            lo, hi = q0 - 0.5 * s, q0 + 0.5 * s
            if self.thinc_on and (v < self.N - 1 or v == self.ir):
                tl, th = self.thinc(qm, q0, qp, lo, hi)
                tbv = lambda x, y: ((at(y, 0, n + 2) - at(x, 1, n + 2)).abs() +  # noqa: E731
                                    (at(y, 1, n + 2) - at(x, 2, n + 2)).abs())
                use = tbv(tl, th) < tbv(lo, hi)                                # cells -1 .. n
                lo = torch.where(use, at(tl, 1, n + 2), at(lo, 1, n + 2))
                hi = torch.where(use, at(th, 1, n + 2), at(hi, 1, n + 2))
            else:
                lo, hi = at(lo, 1, n + 2), at(hi, 1, n + 2)
            L.append(at(hi, 0, n + 1))
            R.append(at(lo, 1, n + 1))
        return L, R

    def flux(self, d, wL, wR):
        """HLLC; returns the fluxes, u*_d and the row V*_db."""
        l, r = self.state(wL), self.state(wR)
        uL, uR = l["u"][d], r["u"][d]
        H = lambda s, a: 2 * s["G"] * s["H"][(a, d)] if self.nv else torch.zeros_like(s["p"])  # noqa: E731
        TL, TR = l["p"] - H(l, d), r["p"] - H(r, d)
        SL, SR = torch.minimum(uL - l["c"], uR - r["c"]), torch.maximum(uL + l["c"], uR + r["c"])
        Ss = ((TR - TL + l["rho"] * uL * (SL - uL) - r["rho"] * uR * (SR - uR)) /
              (l["rho"] * (SL - uL) - r["rho"] * (SR - uR)))
        left = (SL >= 0) | (Ss >= 0)
        star = ~(SL >= 0) & ((Ss >= 0) | (SR > 0))
        K = lambda a, b: torch.where(left, a, b)  # noqa: E731
        up = lambda a, b: torch.where(Ss > 0, a, torch.where(Ss < 0, b, 0.5 * (a + b)))  # noqa: E731
        S, T, rho, E, un = K(SL, SR), K(TL, TR), K(l["rho"], r["rho"]), K(l["rhoE"], r["rhoE"]), K(uL, uR)
        chi = torch.where(star, (S - un) / torch.where(star, S - Ss, 1.0), 0.0)
        F = [None] * self.nvar
        carried = [(self.iar + k, K(l["ar"][k], r["ar"][k])) for k in range(self.N)]
        if self.p.history:
            carried += [(self.ih + k, K(l["ar"][k] * l["eps"][k], r["ar"][k] * r["eps"][k])) for k in range(self.N)]
        for v, m in carried:
            F[v] = m * un + torch.where(star, S * (m * chi - m), 0.0)
        ZL, ZR = torch.sqrt(l["rho"] * l["G"]), torch.sqrt(r["rho"] * r["G"])
        Z = ZL + ZR
        stiff, Zs = Z > 0, torch.where(Z > 0, Z, 1.0)
        work, work_s, us = T * un, 0.0, []
        for a in range(self.dim):
            u = K(l["u"][a], r["u"][a])
            m = rho * u
            if a == d:
                F[self.iu + a] = m * un + T + torch.where(star, S * (rho * chi * Ss - m), 0.0)
                us.append(torch.where(star, Ss, un))
                continue
            sL, sR = H(l, a), H(r, a)
            sig = torch.where(stiff, (ZR * sL + ZL * sR + ZL * ZR * (r["u"][a] - l["u"][a])) / Zs, 0.0)
            ut = torch.where(stiff, (ZL * l["u"][a] + ZR * r["u"][a] + sR - sL) / Zs, up(l["u"][a], r["u"][a]))
            F[self.iu + a] = m * un + torch.where(star, S * (rho * chi * u - m) - sig, -K(sL, sR))
            work_s = work_s + torch.where(star, -ut * sig, -u * K(sL, sR))
            us.append(torch.where(star, ut, u))
        Es = rho * chi * (E / rho + (Ss - un) * (Ss + T / (rho * (S - un))))
        F[self.iE] = E * un + work + work_s + torch.where(star, S * (Es - E), 0.0)
        for k in range(self.N - 1):
            F[k] = up(l["phi"][k], r["phi"][k]) * us[d]
        V = [up(wL[self.iv + k], wR[self.iv + k]) for k in range(self.nv)]
        row = {b: V[k] for k, (a, b) in enumerate(self.vmap) if a == d}
        for k, (a, b) in enumerate(self.vmap):
            F[self.iv + k] = V[k] * us[d]
            if a < self.dim and b in row:
                F[self.iv + k] = F[self.iv + k] - row[b] * us[a]
        F[self.ir] = (wL[self.ir] if self.v[d] > 0 else wR[self.ir]) * self.v[d]
        return F, us[d], row

    def D(self, U):
        w = self.to_prim(U)
        out = [torch.zeros_like(q) for q in U]
        for d in range(self.dim):
            F, us, row = self.flux(d, *self.faces(d, w))
            dif = lambda q: q.diff(dim=3 - d) / self.dx[d]  # noqa: E731
            du = dif(us)
            for v in range(self.nvar):
                out[v] += dif(F[v])
                if v < self.N - 1:
                    out[v] -= w[v] * du
                if self.iv <= v < self.iv + self.nv:
                    a, b = self.vmap[v - self.iv]
                    out[v] -= 2.0 / 3 * w[v] * du
                    if a < self.dim and b in row:
                        out[v] += w[self.iu + a] * dif(row[b])
        return out

    # ---- rigid body
    def gradient(self, r):
        g = []
        for d in range(self.dim):
            i = torch.arange(self.n[d], device=self.dev)
            n = self.n[d]
            hi, lo = ((i + 1) % n, (i - 1) % n) if self.p.periodic[d] else ((i + 1).clamp_max(n - 1), (i - 1).clamp_min(0))
            g.append((r.index_select(3 - d, hi) - r.index_select(3 - d, lo)) / (2 * self.dx[d]))
        return g

    def seed(self):
        r, dxm = self.U[self.ir], min(self.dx)
        g = self.gradient(r)
        gn = torch.sqrt(sum(a * a for a in g))
        band = ((r > 0.5) & (gn * dxm > 1e-10)).nonzero(as_tuple=True)
        if not band[0].numel():
            return
        nrm = [-a[band] / gn[band] for a in g]
        cell = [band[3 - d] for d in range(self.dim)]
        found = torch.zeros(band[0].shape, dtype=torch.bool, device=self.dev)
        wint = [torch.zeros(band[0].shape, dtype=torch.float64, device=self.dev) for _ in range(self.nvar)]
        W = self.to_prim(self.U)
        for step in range(7):
            dist = (1 + 0.5 * step) * dxm
            base, frac = [], []
            for d in range(self.dim):
                xc = self.p.lo[d] + (cell[d].double() + 0.5) * self.dx[d]
                fi = (xc + dist * nrm[d] - self.p.lo[d]) / self.dx[d] - 0.5
                fl = fi.floor()
                f = fi - fl
                up = f > 1 - 1e-3
                base.append((fl + up).long())
                frac.append(torch.where(up | (f < 1e-3), 0.0, f))
            ok, val = ~found, [torch.zeros_like(q) for q in wint]
            for m in range(1 << self.dim):
                idx, wt, inside = [band[0]], 1.0, torch.ones_like(found)
                for d in range(self.dim):
                    ii = base[d] + ((m >> d) & 1)
                    if self.p.periodic[d]:
                        ii = ii % self.n[d]
                    else:
                        inside = inside & (ii >= 0) & (ii < self.n[d])
                    wt = wt * (frac[d] if (m >> d) & 1 else 1 - frac[d])
                    idx.insert(1, ii.clamp(0, self.n[d] - 1))
                while len(idx) < 4:
                    idx.insert(1, torch.zeros_like(band[0]))
                idx = tuple(idx)
                ok = ok & ((wt <= 0) | (inside & (r[idx] < 0.5)))
                val = [a + torch.where(wt > 0, wt * q[idx], 0.0) for a, q in zip(val, W)]
            wint = [torch.where(ok, a, q) for a, q in zip(val, wint)]
            found = found | ok
        keep = found.nonzero(as_tuple=True)[0]
        band, nrm, w = tuple(i[keep] for i in band), [a[keep] for a in nrm], [q[keep] for q in wint]
        nrm += [torch.zeros_like(nrm[0])] * (3 - self.dim)
        P = [[(1.0 if a == b else 0.0) - 2 * nrm[a] * nrm[b] for b in range(3)] for a in range(3)]
        vn = sum(self.v[a] * nrm[a] for a in range(3))
        u = [w[self.iu + a] for a in range(self.dim)]
        for a in range(self.dim):
            w[self.iu + a] = 2 * vn * nrm[a] + sum(P[a][b] * u[b] for b in range(self.dim))
        if self.nv:
            A = [[0.0] * 3 for _ in range(3)]
            for k, (a, b) in enumerate(self.vmap):
                A[a][b] = w[self.iv + k]
            PA = [[sum(P[a][m] * A[m][b] for m in range(3)) for b in range(3)] for a in range(3)]
            for k, (a, b) in enumerate(self.vmap):
                w[self.iv + k] = sum(PA[a][m] * P[m][b] for m in range(3))
        w[self.ir] = r[band]
        for v, q in enumerate(self.to_cons(w)):
            if v != self.ir:
                self.U[v] = self.U[v].index_put(band, q)

    # ---- plasticity
    def yield_stress(self, s, rate):
        num = den = 0.0
        for l, m in enumerate(self.p.mats):
            Gam, _, pr, _, _, _ = self.ref(m, s["rl"][l], s["J2"])
            sy = torch.full_like(s["p"], m.get("sigY", 0.0))
            if m.get("jc_c1"):
                T = 298.0 + (s["p"] - pr) / (s["rl"][l] * Gam * m["jc_cv"])
                ts = ((T - 298.0) / (m["jc_tmelt"] - 298.0)).clamp(0, 1)
                eps = s["eps"][l].clamp_min(0) if s["eps"] else torch.zeros_like(T)
                sy = ((m["jc_c1"] + m["jc_c2"] * eps ** m["jc_n"]) *
                      (1 + m["jc_c3"] * torch.log(torch.clamp_min(rate, 1.0))) * (1 - ts ** m["jc_m"]))
            num, den = num + s["phi"][l] * sy / Gam, den + s["phi"][l] / Gam
        return num / den

    def plastic(self, U, dt, rigid):
        s = self.state(self.to_prim(U))
        nd = s["J2"].sqrt()
        svm = math.sqrt(1.5) * 2 * s["G"] * nd
        sy = s["sigY"]
        if any(m.get("jc_c1") for m in self.p.mats):
            zero = torch.zeros_like(svm)
            sy0 = self.yield_stress(s, zero)
            over = svm > sy0
            rate = torch.where(over, math.sqrt(2.0 / 3) * (1 - sy0 / torch.where(over, svm, 1.0)) * nd / dt, zero)
            sy = self.yield_stress(s, rate)
        over = svm > sy
        sc = torch.where(over, sy / torch.where(over, svm, 1.0), 1.0)
        e = [torch.exp(sc * d) for d in s["d"]]
        av, df = 0.5 * (e[0] + e[1]), 0.5 * (e[0] - e[1])
        A = [av + df * s["c2a"], df * s["s2a"], df * s["s2a"], av - df * s["c2a"], e[2]]
        U = list(U)
        for k in range(self.nv):
            U[self.iv + k] = torch.where(rigid, U[self.iv + k], A[k])
        if self.p.history:
            deps = torch.where(rigid, 0.0, math.sqrt(2.0 / 3) * (1 - sc) * nd)
            for l, m in enumerate(self.p.mats):
                if m.get("sigY") or m.get("jc_c1"):
                    U[self.ih + l] = U[self.ih + l] + U[self.iar + l] * deps
        return U

    # ---- time
    def step(self):
        s = self.state(self.to_prim(self.U))
        speed = sum((u.abs() + s["c"]) / self.dx[d] for d, u in enumerate(s["u"])).amax(dim=(1, 2, 3))
        speed = speed.clamp_min(sum(abs(self.v[d]) / self.dx[d] for d in range(self.dim)))
        dt = (self.p.cfl / speed).reshape(-1, 1, 1, 1)
        self.seed()
        if self.p.dynamic:
            pr, dV = self.to_prim(self.U)[self.iE], math.prod(self.dx)
            self.force = [float((pr * g).sum() * dV) for g in self.gradient(self.U[self.ir])] + [0.0] * (3 - self.dim)
        Un = self.U
        rigid = Un[self.ir] > 0.5

        def stage(U, ca, cb):
            D = self.D(U)
            new = [ca * a + cb * (q - dt * x) for a, q, x in zip(Un, U, D)]
            return [q if v == self.ir else torch.where(rigid, a, q) for v, (a, q) in enumerate(zip(Un, new))]

        U = stage(stage(stage(Un, 0.0, 1.0), 0.75, 0.25), 1.0 / 3, 2.0 / 3)
        if self.nv:
            U = self.plastic(U, dt, rigid)
        self.U = U
        self.t = self.t + dt
        if self.p.dynamic:
            h = float(dt)
            self.v = [a + h * f / self.p.mass for a, f in zip(self.v, self.force)]
            self.x = [a + h * v for a, v in zip(self.x, self.v)]


def exact(case, seed):
    """The pass in 64 bits, laid out as run() returns it."""
    dev = torch.device("cuda:0" if torch.cuda.is_available() else "cpu")
    ps = _problems(case, seed, dev)
    if case["flow"] == "batch":
        parts = [None] * len(ps)
        for n in sorted({p.n for p in ps}):
            at = [i for i, p in enumerate(ps) if p.n == n]
            for k in range(0, len(at), 16):
                e = _Exact([ps[i] for i in at[k:k + 16]], True)
                for _ in range(case["steps"]):
                    e.step()
                for j, i in enumerate(at[k:k + 16]):
                    parts[i] = torch.cat([q[j].reshape(-1) for q in e.U])
        return torch.cat(parts)
    p = ps[0]
    e = _Exact(ps, case.get("thinc", True))
    for _ in range(case["steps"]):
        e.step()
    out = _groups(p, torch.stack([q.reshape(-1) for q in e.U]))
    out["time"] = float(e.t)
    if p.dynamic:
        out.update(_body(case, p, *(np.array(a) for a in (e.force, e.v, e.x))))
    return out
