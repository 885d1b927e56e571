"""What this framework's speed is measured on: the calls its users make, over the sizes they make
them at.

listed() names the cases, draw(rng) gives more of the same ranges, prepare(case, seed) builds what a
program holds before the call (the lattice with its parameters and its initial densities, output
buffers), run(state) makes one pass through the package's public entry points, work(case) is what a
pass cannot do without, and exact(case, seed) the same results in 64 bits, written here in plain
torch from the model's equations.

Four kinds of pass:
  flow      a two-dimensional run advanced by `steps` time steps, its populations exported; with
            `observe` = k every k-th step is sampled and the time averages are read at the end
  sweep     the same for a batch of channels of different heights and body forces in one lattice
  gradient  J, dJ/drho and dJ/dtheta of a run of `steps` steps through the discrete adjoint
  flow3     a three-dimensional run, its fields read; with `totals` every step's mass and momentum

A flow goes on from where the pass before left it, as a simulation does.  Results of an FP32 lattice
are kept in float32, the precision they have; those of an FP64 lattice in float64.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint as recompute

from paper_1402_6019_gb300 import adjoint
from paper_1402_6019_gb300 import lbm as L

THIRD = 1.0 / 3.0
PRECISION = {"f32": L.LBM_FP32, "f64": L.LBM_FP64}
DTYPE = {"f32": torch.float32, "f64": torch.float64}

# Couplings: the two-species emulsion, the single-component fluid of the noise runs, and the
# phase-separating film couplings of the droplet runs.
FLUIDS = {
    "emulsion": dict(ns=2, G1=(-9.0, -8.0), G2=(8.1, 7.1), G_AB=0.405, rho0=0.83, rho=(1.2, 0.05)),
    "single": dict(ns=1, G1=(-9.0, -9.0), G2=(8.1, 8.1), G_AB=0.0, rho0=1.0, rho=None),
    "film": dict(ns=1, G1=(-20.4, -20.4), G2=(16.0, 16.0), G_AB=0.0, rho0=1.0, rho=(1.39, 0.285)),
}
SWEEP_DRIVES = (1e-6, 3e-6, 1e-5)


def flow(nx, nz, fluid="emulsion", precision="f32", walls=False, drive="none", steps=32, observe=0, tau=1.0):
    return dict(kind="flow", nx=nx, nz=nz, fluid=fluid, precision=precision, walls=walls, drive=drive, steps=steps,
                observe=observe, tau=tau)


def sweep(nx, low, high, by, precision="f32", steps=8, observe=1):
    return dict(kind="sweep", nx=nx, low=low, high=high, by=by, precision=precision, steps=steps, observe=observe)


def gradient(nx, nz, precision="f32", fluid="emulsion", steps=200, every=25):
    return dict(kind="gradient", nx=nx, nz=nz, precision=precision, fluid=fluid, steps=steps, every=every)


def flow3(nx, ny, nz, precision="f32", fluid="emulsion", walls=False, steps=20, totals=False):
    return dict(kind="flow3", nx=nx, ny=ny, nz=nz, precision=precision, fluid=fluid, walls=walls, steps=steps,
                totals=totals)


def listed():
    return [
        # The small single-component lattice of the noise runs, stepped in FP64 without sampling:
        # every step is a small launch, so what a launch and its latency cost shows here.
        dict(flow(128, 128, "single", "f64", steps=100), name="noise_128_f64"),
        # A droplet in its vapour (Laplace's law), FP64, a size that no tile divides.
        dict(flow(201, 173, "film", "f64", steps=50, observe=0), name="droplet_201x173_f64"),
        # A small emulsion watched every step.
        dict(flow(256, 256, steps=100, observe=1), name="emulsion_256_observed"),
        # The benchmarked emulsion, FP32, every step sampled.
        dict(flow(1024, 1024, steps=32, observe=1), name="emulsion_1024_observed"),
        # The large emulsion, stepped without sampling between two looks at it.
        dict(flow(4096, 4096, steps=8), name="emulsion_4096"),
        # The sheared channel, relaxation times off 1, sampled now and then, as rheology runs do.
        dict(flow(2048, 256, walls=True, drive="couette", steps=50, observe=10, tau=0.9), name="couette_2048x256"),
        # The channel under a body force in FP64: the reference that FP32 results are held against.
        dict(flow(2048, 256, precision="f64", walls=True, drive="poiseuille", steps=6, observe=1),
             name="poiseuille_2048x256_f64"),
        # The width and drive sweep: 48 channels of 32 .. 512 rows in one lattice, every step sampled.
        dict(sweep(1024, 32, 512, 32, steps=8), name="sweep_48"),
        # Calibration: the gradient of a run on the 256 x 256 emulsion, snapshots every 25 steps.
        dict(gradient(256, 256, steps=200), name="gradient_256"),
        # The same in FP64 on a ragged lattice, a run that ends inside a segment.
        dict(gradient(150, 90, "f64", steps=60), name="gradient_150x90_f64"),
        # The three-dimensional emulsion.
        dict(flow3(128, 128, 128, steps=20), name="emulsion3d_128"),
        # A three-dimensional channel in FP64, odd sizes, its totals followed every step.
        dict(flow3(65, 48, 33, "f64", walls=True, steps=8, totals=True), name="channel3d_65x48x33_f64"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("flow", "flow", "flow", "sweep", "gradient", "flow3"))
    precision = rng.choice(("f32", "f32", "f64"))
    slow = 16 if precision == "f64" else 1  # an FP64 step costs that much more
    if kind == "flow":
        walls = rng.random() < 0.4
        nx, nz = log(96, 4096), log(40 if walls else 96, 2048)
        sites = nx * nz * slow
        return flow(nx, nz, "emulsion" if rng.random() < 0.7 else rng.choice(("single", "film")), precision, walls,
                    rng.choice(("couette", "poiseuille")) if walls else "none",
                    max(4, min(100, 100_000_000 // sites)), rng.choice((0, 1, 1, 7)), rng.choice((1.0, 1.0, 0.8)))
    if kind == "sweep":
        by = rng.choice((16, 24, 37))
        return sweep(log(200, 1500), by, by * rng.randint(3, 10), by, "f32", rng.randint(4, 10), rng.choice((0, 1)))
    if kind == "gradient":
        nx, nz = log(60, 400), log(60, 300)
        return gradient(nx, nz, precision, "emulsion" if rng.random() < 0.7 else "single",
                        max(10, min(120, 12_000_000 // (nx * nz * (4 if precision == "f64" else 1)))),
                        rng.choice((10, 25)))
    nx, ny, nz = log(40, 160), log(24, 130), log(24, 130)
    return flow3(nx, ny, nz, precision, "emulsion" if rng.random() < 0.7 else "film", rng.random() < 0.4,
                 max(3, min(24, 30_000_000 // (nx * ny * nz * slow))), rng.random() < 0.4)


# ---- inputs ---------------------------------------------------------------------------------

def _runs(rows, start, length, n_rows, nx):
    """Sites covered by runs of `length` sites from `start` (periodic) in the given rows: bool [n_rows, nx]."""
    rows, start = torch.from_numpy(rows).cuda(), torch.from_numpy(start).cuda()
    length = torch.from_numpy(np.minimum(length, nx)).cuda()
    start = torch.remainder(start, nx)
    end = start + length
    edge = torch.zeros(n_rows * (2 * nx + 1), dtype=torch.int32, device="cuda")
    one = torch.ones_like(rows, dtype=torch.int32)
    edge.index_add_(0, rows * (2 * nx + 1) + start, one)
    edge.index_add_(0, rows * (2 * nx + 1) + end, -one)
    inside = edge.view(n_rows, 2 * nx + 1).cumsum(1) > 0
    return inside[:, :nx] | inside[:, nx:2 * nx]


def _disks(nx, nz, fraction, rng, r_mean=12.0, r_spread=3.0, periodic_z=True):
    """Overlapping disks of radius r_mean +- r_spread, as many as cover `fraction` of the lattice: bool [nz, nx]."""
    r_mean = min(r_mean, 0.2 * min(nx, nz))
    r_spread = min(r_spread, 0.3 * r_mean)
    n = max(1, math.ceil(-math.log(1.0 - fraction) * nx * nz / (math.pi * (r_mean ** 2 + r_spread ** 2 / 3))))
    cx, cz = rng.uniform(0, nx, n), rng.uniform(0, nz, n)
    r = r_mean + r_spread * rng.uniform(-1, 1, n)
    d = np.arange(-math.ceil(r_mean + r_spread), math.ceil(r_mean + r_spread) + 1)
    z = np.floor(cz)[:, None].astype(np.int64) + d
    w2 = r[:, None] ** 2 - (z - cz[:, None]) ** 2
    ok = w2 >= 0
    if not periodic_z:
        ok &= (z >= 0) & (z < nz)
    w = np.sqrt(np.where(ok, w2, 0.0))
    x0 = np.ceil(cx[:, None] - w).astype(np.int64)
    x1 = np.floor(cx[:, None] + w).astype(np.int64)
    ok &= x1 >= x0
    return _runs((z % nz)[ok], x0[ok], (x1 - x0 + 1)[ok], nz, nx)


def _spheres(nx, ny, nz, fraction, rng, r_mean=8.0, r_spread=2.0, periodic_z=True):
    """The same with spheres: bool [nz, ny, nx]."""
    r_mean = min(r_mean, 0.2 * min(nx, ny, nz))
    r_spread = min(r_spread, 0.3 * r_mean)
    volume = 4.0 / 3.0 * math.pi * (r_mean ** 3 + r_mean * r_spread ** 2)
    n = max(1, math.ceil(-math.log(1.0 - fraction) * nx * ny * nz / volume))
    cx, cy, cz = rng.uniform(0, nx, n), rng.uniform(0, ny, n), rng.uniform(0, nz, n)
    r = r_mean + r_spread * rng.uniform(-1, 1, n)
    d = np.arange(-math.ceil(r_mean + r_spread), math.ceil(r_mean + r_spread) + 1)
    y = (np.floor(cy)[:, None].astype(np.int64) + d)[:, None, :]
    z = (np.floor(cz)[:, None].astype(np.int64) + d)[:, :, None]
    w2 = r[:, None, None] ** 2 - (y - cy[:, None, None]) ** 2 - (z - cz[:, None, None]) ** 2
    ok = w2 >= 0
    if not periodic_z:
        ok &= (z >= 0) & (z < nz)
    w = np.sqrt(np.where(ok, w2, 0.0))
    x0 = np.ceil(cx[:, None, None] - w).astype(np.int64)
    x1 = np.floor(cx[:, None, None] + w).astype(np.int64)
    ok &= x1 >= x0
    row = np.broadcast_to((z % nz) * ny + y % ny, w.shape)
    return _runs(row[ok], x0[ok], (x1 - x0 + 1)[ok], nz * ny, nx).view(nz, ny, nx)


def _densities(case, seed):
    """rho [ns, (nz,) ny or nz, nx], FP64 on the GPU."""
    rng = np.random.RandomState(seed % (1 << 32))
    if case["kind"] == "sweep":
        parts = [_disks(case["nx"], h, 0.85, rng, periodic_z=False) for h in _heights(case)]
        inside = torch.cat(parts)
        return _two_phases(inside, 2, FLUIDS["emulsion"]["rho"])
    fluid = FLUIDS[case["fluid"]]
    if case["kind"] == "flow3":
        if fluid["rho"] is None:
            return _noise((fluid["ns"], case["nz"], case["ny"], case["nx"]), seed)
        inside = _spheres(case["nx"], case["ny"], case["nz"], 0.5, rng, periodic_z=not case["walls"])
        return _two_phases(inside, fluid["ns"], fluid["rho"])
    if fluid["rho"] is None:
        return _noise((fluid["ns"], case["nz"], case["nx"]), seed)
    walls = bool(case.get("walls"))
    if case["fluid"] == "film":  # droplets of the liquid in its vapour
        inside = _disks(case["nx"], case["nz"], 0.3, rng, r_mean=24.0, r_spread=6.0, periodic_z=not walls)
    else:
        inside = _disks(case["nx"], case["nz"], 0.85 if walls else 0.8, rng, periodic_z=not walls)
    return _two_phases(inside, fluid["ns"], fluid["rho"])


def _noise(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return 1.0 + 0.01 * (2.0 * torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") - 1.0)


def _two_phases(inside, ns, rho):
    a = torch.where(inside, rho[0], rho[1]).double()
    return torch.stack([a, torch.where(inside, rho[1], rho[0]).double()]) if ns == 2 else a[None].contiguous()


def _heights(case):
    return [h for h in range(case["low"], case["high"] + 1, case["by"]) for _ in SWEEP_DRIVES]


def _targets(case, seed):
    """The profiles that a calibration aims at: a velocity of the order the drive reaches, a density between the phases'."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    t = torch.rand((2, case["nz"]), generator=g, dtype=torch.float64, device="cuda")
    return 1e-3 * t[0], 0.3 + 0.6 * t[1]


def _params(case):
    fluid = FLUIDS[case.get("fluid", "emulsion")]
    tau = case.get("tau", 1.0)
    p = dict(tau=(tau, tau), G1=fluid["G1"], G2=fluid["G2"], G_AB=fluid["G_AB"], rho0=(fluid["rho0"],) * 2,
             weight_norm=THIRD)
    if case.get("drive") == "couette" or (case["kind"] == "flow3" and case["walls"]):
        p["wall_u"] = (-0.01, 0.01)
    if case.get("drive") == "poiseuille":
        p["body_force"] = 1e-6
    if case["kind"] == "gradient":
        p["body_force"] = 1e-5
    return p


# ---- the measured pass ------------------------------------------------------------------------

class State:
    pass


_streams = []


def _stream():
    """The program's stream: its lattices and its torch work follow one another on it."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    with torch.cuda.stream(_stream()):
        return _prepare(case, seed)


def _prepare(case, seed):
    s = State()
    s.case, s.dtype = case, DTYPE[case["precision"]]
    rho = _densities(case, seed)
    s.ns = rho.shape[0]
    prec = PRECISION[case["precision"]]
    stream = _stream().cuda_stream
    if case["kind"] == "flow3":
        s.lat = L.Lattice3(case["nx"], case["ny"], case["nz"], s.ns, prec, int(case["walls"]), stream=stream,
                         **_params(case))
        s.lat.set_fields(rho)
        shape = tuple(rho.shape[1:])
        s.rho = torch.empty((s.ns,) + shape, dtype=torch.float64, device="cuda")
        s.u = torch.empty((3,) + shape, dtype=torch.float64, device="cuda")
        s.f = torch.empty((s.ns, 19) + shape, dtype=torch.float64, device="cuda")
        s.totals = torch.empty((case["steps"], 5), dtype=torch.float64, device="cuda")
        return s
    if case["kind"] == "sweep":
        heights = _heights(case)
        s.lat = L.Lattice(case["nx"], None, 2, prec, L.LBM_BOUNCEBACK, instances=heights, stream=stream,
                        **_params(case))
        for i in range(len(heights)):
            s.lat.set_instance_drive(i, SWEEP_DRIVES[i % len(SWEEP_DRIVES)], (0.0, 0.0))
    else:
        s.lat = L.Lattice(case["nx"], case["nz"], s.ns, prec, int(bool(case.get("walls"))), stream=stream,
                        **_params(case))
    if case["kind"] == "gradient":
        s.rho = rho
        s.target_u, s.target_rho = _targets(case, seed)
        return s
    s.lat.set_fields(rho)
    s.lat.set_observe(case["observe"])
    s.f = torch.empty((s.ns, 9) + tuple(rho.shape[1:]), dtype=s.dtype, device="cuda")
    return s


def run(s):
    with torch.cuda.stream(_stream()):
        return _run(s)


def _run(s):
    case = s.case
    if case["kind"] == "gradient":
        J, g_rho, g_theta = adjoint.rollout_gradient(s.lat, s.rho, case["steps"], s.target_u, s.target_rho,
                                                     checkpoint=case["every"])
        return {"J": J, "rho": g_rho.to(s.dtype), "theta": g_theta.to(s.dtype)}
    if case["kind"] == "flow3":
        if case["totals"]:
            s.lat.step_totals(case["steps"], s.totals)
        else:
            s.lat.step(case["steps"])
        p = [ctypes.c_void_p(t.data_ptr()) for t in (s.rho, s.u, s.f)]
        rc = L.load().lbm3_get_fields(s.lat.h, *p, L.LBM_DEVICE)  # waits for the lattice's stream
        if rc != L.LBM_OK:
            raise L.LbmError(rc, "lbm3_get_fields")
        out = {"rho": s.rho, "u": s.u, "f": s.f}
        if case["totals"]:
            out["totals"] = s.totals
        return {k: v.to(s.dtype) for k, v in out.items()}
    s.lat.step(case["steps"])
    L.lbm_export_state(s.lat.h, s.f)
    out = {"f": s.f}
    if case["observe"]:
        # the averages of what was sampled; the fluidity, a ratio of two profiles that are near zero
        # over so few steps, is formed from long averages only
        a = s.lat.averages(reset=True)
        kind = np.float32 if case["precision"] == "f32" else np.float64
        out["across"] = np.concatenate([a["ux_z"][None], a["rho_z"], a["sxz_z"][None]]).astype(kind)
        out["along"] = np.stack([a["ps_x"], a["pxx_x"]]).astype(kind)
        out["mass"] = a["mass"].astype(kind)
    return out


def work(case):
    """Each population read and written once a step; the operations of the model at a site (moments,
    pseudopotential, the force's differences, collision) counted once."""
    size = 4 if case["precision"] == "f32" else 8
    if case["kind"] == "flow3":
        ns, sites, q, per_site = FLUIDS[case["fluid"]]["ns"], case["nx"] * case["ny"] * case["nz"], 19, 420
    elif case["kind"] == "sweep":
        ns, sites, q, per_site = 2, case["nx"] * sum(_heights(case)), 9, 190
    else:
        ns, sites, q, per_site = FLUIDS[case["fluid"]]["ns"], case["nx"] * case["nz"], 9, 190
    if case["kind"] == "gradient":
        # forward; forward again with the states kept; back: state and adjoint read, adjoint written
        moved, ops = 2 + 3 + 3, 2 * per_site + 500
    else:
        moved, ops = 2, per_site + (120 / max(1, case["observe"]) if case.get("observe") else 0)
    return {"bytes": float(case["steps"]) * sites * ns * q * size * moved, "flops": float(case["steps"]) * sites * ns * ops}


# ---- the same in 64 bits ------------------------------------------------------------------------

C9 = ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP9 = (0, 3, 4, 1, 2, 7, 8, 5, 6)
ATT2, REP2, BELT2 = {1: 4 / 15, 2: 1 / 10, 4: 1 / 120}, {1: 4 / 21, 2: 4 / 45, 4: 1 / 60, 5: 2 / 315, 8: 1 / 5040}, {1: 1 / 3, 2: 1 / 12}
C19 = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
       (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1))
W19 = (1 / 3,) + (1 / 18,) * 6 + (1 / 36,) * 12
OPP19 = (0,) + tuple(l + 1 if l % 2 else l - 1 for l in range(1, 19))
ATT3, REP3, BELT3 = ({1: 2 / 15, 2: 1 / 15, 3: 1 / 60, 4: 1 / 120},
                     {1: 4 / 45, 2: 1 / 21, 3: 2 / 105, 4: 5 / 504, 5: 1 / 315, 6: 1 / 630, 8: 1 / 5040}, {1: 1 / 6, 2: 1 / 12})


class Model:
    """The step of one lattice, dims = (nz, nx) or (nz, ny, nx), on FP64 tensors."""

    def __init__(self, params, ns, dims, walls):
        self.ns, self.dims, self.walls, self.p = ns, dims, walls, params
        two = len(dims) == 2
        self.C, self.W, self.opp = (C9, W9, OPP9) if two else (C19, W19, OPP19)
        self.att, self.rep, self.belt = (ATT2, REP2, BELT2) if two else (ATT3, REP3, BELT3)
        shape = (ns,) + (1,) * len(dims)

        def col(v):
            return torch.tensor(v[:ns], dtype=torch.float64, device="cuda").view(shape)

        self.tau, self.G1, self.G2 = col(params["tau"]), col(params["G1"]), col(params["G2"])
        self.G_AB = torch.tensor(params["G_AB"], dtype=torch.float64, device="cuda")
        self.g = torch.tensor(params.get("body_force", 0.0), dtype=torch.float64, device="cuda")
        self.rho0, self.wall_u = params["rho0"][0], params.get("wall_u", (0.0, 0.0))
        r = range(-2, 3)
        # offsets (dx, [dy,] dz) of the interaction links
        links = [(x, z) for z in r for x in r] if two else [(x, y, z) for z in r for y in r for x in r]
        self.links = [c for c in links if 0 < sum(v * v for v in c) <= 8]
        self.index = []
        for axis, n in enumerate(dims):
            i = np.arange(-2, n + 2)
            if axis == 0 and walls:  # mirror images beyond the walls at -1/2 and n - 1/2
                m = i % (2 * n)
                i = np.where(m >= n, 2 * n - 1 - m, m)
            self.index.append(torch.from_numpy(i % n).cuda())

    def window(self, a):
        """shift(c)(x) = a(x + c), |c_i| <= 2."""
        for axis, i in enumerate(self.index):
            a = a.index_select(axis + 1, i)

        def shift(c):
            at = tuple(slice(2 + d, 2 + d + n) for d, n in zip(reversed(c), self.dims))
            return a[(slice(None),) + at]

        return shift

    def start(self, rho):
        return torch.stack([w * rho for w in self.W], dim=1)

    def moments(self, f):
        rho = f.sum(1)
        j = [sum(f[:, l] * c[d] for l, c in enumerate(self.C) if c[d]) for d in range(len(self.dims))]
        return rho, j

    def force(self, rho, psi, rs):
        """Per species and direction, x first."""
        ps = self.window(psi)
        att, rep = [0.0] * len(self.dims), [0.0] * len(self.dims)
        for c in self.links:
            q = sum(v * v for v in c)
            v = ps(c)
            for d in range(len(c)):
                if c[d]:
                    att[d] = att[d] + self.att.get(q, 0.0) * c[d] * v if q in self.att else att[d]
                    rep[d] = rep[d] + self.rep[q] * c[d] * v
        n = self.p["weight_norm"]
        F = [-n * psi * (self.G1 * a + self.G2 * r) for a, r in zip(att, rep)]
        if self.ns == 2:
            for d in range(len(self.dims)):
                x = sum(self.belt[sum(v * v for v in c)] * c[d] * rs(c).flip(0) for c in self.links
                        if sum(v * v for v in c) <= 2 and c[d])
                F[d] = F[d] - n * self.G_AB * rho * x
        F[0] = F[0] + rho * self.g
        return F, ps

    def step(self, f, sample=None):
        rho, j = self.moments(f)
        psi = 1.0 - torch.exp(-rho / self.rho0)
        rs = self.window(rho)
        F, ps = self.force(rho, psi, rs)
        den = (rho / self.tau).sum(0)
        u = [((v / self.tau).sum(0) / den) + self.tau * w / rho for v, w in zip(j, F)]
        usq = sum(v * v for v in u)
        if sample is not None:
            self.sample(sample, f, rho, j, F, u, ps, rs, psi)
        g = []
        for l, c in enumerate(self.C):
            cu = sum(c[d] * u[d] for d in range(len(c)) if c[d])
            feq = self.W[l] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)
            g.append(f[:, l] - (f[:, l] - feq) / self.tau)
        new = []
        for l, c in enumerate(self.C):
            v = torch.roll(g[l], tuple(reversed(c)), tuple(range(1, len(c) + 1)))
            if self.walls and c[-1]:  # what comes from beyond a wall: the site's own, reflected
                row, uw = (0, self.wall_u[0]) if c[-1] > 0 else (self.dims[0] - 1, self.wall_u[1])
                v = v.clone()
                v[:, row] = g[self.opp[l]][:, row] + 6.0 * self.W[l] * rho[:, row] * c[0] * uw
            new.append(v)
        return torch.stack(new, dim=1)

    def sample(self, into, f, rho, j, F, u, ps, rs, psi):
        """Adds the observables of the state to `into` (two dimensions)."""
        n = self.p["weight_norm"]
        K = {q: n * (self.G1 * self.att.get(q, 0.0) + self.G2 * w) for q, w in self.rep.items()}
        ux = (j[0] + 0.5 * F[0]).sum(0) / rho.sum(0)
        # interaction stress: node products of the shells 1, 2; 4, 8 with half-link products; 5 with
        # the products of the sites on either side of the link's middle
        comps = []
        for a, b in ((0, 0), (1, 1), (0, 1)):
            s = 0.0
            for c in self.links:
                q, cc = sum(v * v for v in c), c[a] * c[b]
                if not cc:
                    continue
                s = s + (0.5 if q <= 2 else 0.25) * K[q] * cc * psi * ps(c)
                if c[0] < 0 or (c[0] == 0 and c[1] < 0):
                    continue  # one of each antipodal pair
                if q in (4, 8):
                    h = (c[0] // 2, c[1] // 2)
                    s = s + 0.25 * K[q] * cc * 2.0 * ps(h) * ps((-h[0], -h[1]))
                if q == 5:
                    # the four sites around the link centred here: c = m + k, m = first-belt axis, k = diagonal
                    m = (c[0] // 2 if abs(c[0]) == 2 else 0, c[1] // 2 if abs(c[1]) == 2 else 0)
                    k = (c[0] - m[0], c[1] - m[1])
                    s = s + 0.25 * K[q] * cc * (ps(k) * ps((-m[0], -m[1])) + ps(m) * ps((-k[0], -k[1])))
            comps.append(s.sum(0) if torch.is_tensor(s) else torch.zeros_like(ux))
        sxx, szz, sxz = comps
        if self.ns == 2:
            for c in self.links:
                q = sum(v * v for v in c)
                if q > 2:
                    continue
                phi = 0.5 * n * self.G_AB * self.belt[q] * (rho[0] * rs(c)[1] + rho[1] * rs(c)[0])
                sxx, szz, sxz = sxx + c[0] ** 2 * phi, szz + c[1] ** 2 * phi, sxz + c[0] * c[1] * phi
        pi = f[:, 5] + f[:, 7] - f[:, 6] - f[:, 8]
        half = 0.5 / self.tau
        kin = ((1.0 - half) * pi + half * rho * u[0] * u[1]).sum(0)
        push = (self.tau - 0.5) ** 2
        pxx = sxx + (rho / 3.0 + push * F[0] ** 2 / rho).sum(0)
        pzz = szz + (rho / 3.0 + push * F[1] ** 2 / rho).sum(0)
        got = {"ux": ux.mean(1), "rho": rho.mean(2), "sxz": -(kin + sxz).mean(1), "ps": (pxx - pzz).sum(0),
               "pxx": pxx.sum(0), "mass": rho.sum((1, 2)), "n": 1}
        for k, v in got.items():
            into[k] = into.get(k, 0) + v


def _exact_flows(case, seed, parts):
    """parts: (params, walls, rows) of each lattice, stacked in z."""
    rho = _densities(case, seed)
    out, samples, z = [], [], 0
    for params, walls, rows in parts:
        m = Model(params, rho.shape[0], (rows, case["nx"]), walls)
        f, got = m.start(rho[:, z:z + rows]), {}
        for k in range(case["steps"]):
            f = m.step(f, got if case["observe"] and k % case["observe"] == 0 else None)
        out.append(f)
        samples.append(got)
        z += rows
    res = {"f": torch.cat(out, dim=2)}
    if case["observe"]:
        n = samples[0]["n"]
        across = [torch.cat([torch.cat([g["ux"][None], g["rho"], g["sxz"][None]]) for g in samples], dim=1) / n]
        along = torch.stack([sum(g["ps"] for g in samples), sum(g["pxx"] for g in samples)]) / (n * z)
        mass = sum(g["mass"] for g in samples) / n
        if rho.shape[0] == 1:
            mass = torch.cat([mass, torch.zeros_like(mass)])
        res.update(across=across[0].cpu().numpy(), along=along.cpu().numpy(), mass=mass.cpu().numpy())
    return res


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "flow":
            return _exact_flows(case, seed, [(_params(case), bool(case["walls"]), case["nz"])])
        if case["kind"] == "sweep":
            parts = [(dict(_params(case), body_force=SWEEP_DRIVES[i % len(SWEEP_DRIVES)]), True, h)
                     for i, h in enumerate(_heights(case))]
            return _exact_flows(case, seed, parts)
        if case["kind"] == "flow3":
            rho = _densities(case, seed)
            m = Model(_params(case), rho.shape[0], tuple(rho.shape[1:]), bool(case["walls"]))
            f, totals = m.start(rho), []
            for _ in range(case["steps"]):
                f = m.step(f)
                r, j = m.moments(f)
                row = torch.zeros(5, dtype=torch.float64, device="cuda")
                row[:m.ns] = r.sum((1, 2, 3))
                row[2:] = torch.stack([v.sum() for v in j])
                totals.append(row)
            r, j = m.moments(f)
            psi = 1.0 - torch.exp(-r / m.rho0)
            F, _ = m.force(r, psi, m.window(r))
            u = torch.stack([(a + 0.5 * b).sum(0) / r.sum(0) for a, b in zip(j, F)])
            out = {"rho": r, "u": u, "f": f}
            if case["totals"]:
                out["totals"] = torch.stack(totals)
            return out
    # the gradient by differentiating the run itself, each step recomputed on the way back
    rho = _densities(case, seed).requires_grad_()
    m = Model(_params(case), rho.shape[0], (case["nz"], case["nx"]), False)
    theta = [m.G1, m.G2, m.G_AB, m.tau, m.g]
    for t in theta:
        t.requires_grad_()
    f = m.start(rho)
    for _ in range(case["steps"]):
        f = recompute(m.step, f, use_reentrant=False)
    r, j = m.moments(f)
    target_u, target_rho = _targets(case, seed)
    J = (((j[0].sum(0) / r.sum(0)).mean(1) - target_u) ** 2 + (r[0].mean(1) - target_rho) ** 2).sum()
    grads = torch.autograd.grad(J, [rho] + theta, allow_unused=True)
    two = [torch.zeros(2, dtype=torch.float64, device="cuda") for _ in range(3)]
    for k, i in enumerate((1, 2, 4)):  # G1, G2, tau, a pair each
        two[k][:m.ns] = grads[i].flatten()
    cross = grads[3] if grads[3] is not None else torch.zeros((), dtype=torch.float64, device="cuda")
    return {"J": float(J), "rho": grads[0],
            "theta": torch.cat([two[0], two[1], cross.view(1), two[2], grads[5].view(1)])}
