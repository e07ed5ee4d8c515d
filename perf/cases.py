"""What a user of the coupled LBM-DEM library has it do, as cases to time.

A case is a dict of plain numbers and texts.  prepare() builds what a user's
program holds before the call (the simulations, already packed, or the host
arrays of a new packing), run() is one pass through the public entry points
(paper_1808_08921_gb300.lbmdem), and exact() is the same pass in plain FP64
torch, written from the equations, without the library.

The library computes the fluid and the sphere velocities in FP32 (its host
arrays are FP64 containers), so those outputs are handed on as FP32; sphere
centres, which it keeps in FP64, stay FP64.  With 16-bit population storage
the fluid's outputs and the forces summed from it are handed on in the
storage's own form: deviations from rest, FP16 scaled by 2^12.  Time loops go on from pass to
pass, as a user's does; a case that starts from a new packing sets it in
run().  The sources are small-amplitude waves, so that a long loop stays in
the regime it started in.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads
from paper_1808_08921_gb300 import lbmdem

STORAGE = {"f32": lbmdem.F32, "bf16": lbmdem.BF16_DEV, "f16": lbmdem.F16_DEV}
RATIO = 0.35625  # R / a of the FCC packings (5.7 / 16 = 11.4 / 32): slightly overlapping spheres


def listed():
    return [
        # the smallest column of the repository: latency and launches are all of it
        dict(name="column_16x16x128", kind="column", a=16, cx=8, cy=1, cz=1, tau=0.8, period=200, steps=64, k=10,
             storage="f32", read="fields"),
        # the saturated chain of the paper's third benchmark: narrow periodic
        # cross-section, Hertz contacts in a line
        dict(name="chain_12x12x620", kind="chain", n=60, steps=64, k=10, mobile=True),
        # a new packing of free spheres per pass, from host arrays: ragged
        # box, fast spheres (nodes converted every step), then the whole state
        dict(name="spheres_61x37x45", kind="spheres", nx=61, ny=37, nz=45, n=24, R=4.5, vel=0.01, steps=48,
             tau=0.7, periodic=False),
        # one sphere settling in a periodic box (the paper's first benchmark):
        # nearly all nodes are fluid, one contact-free sphere
        dict(name="settle_160", kind="settle", L=160, R=5.005, tau=1.0, steps=32),
        # spheres alone, before the fluid is switched on: more of them than
        # the large column has
        dict(name="dry_4096", kind="dry", a=32, cx=64, cy=4, cz=4, k=10, steps=64),
        # 16-bit storage with the probe and the totals recorded, as in the
        # source study's columns
        dict(name="column_bf16_32x32x512", kind="column", a=16, cx=32, cy=2, cz=2, tau=0.8, period=100, steps=32,
             k=2, storage="bf16", read="probe"),
        # the precision configuration: ordinary size, small spheres
        dict(name="column_f32_64x64x512", kind="column", a=16, cx=32, cy=4, cz=4, tau=0.8, period=200, steps=64,
             k=10, storage="f32", read="planes"),
        dict(name="column_f16_64x64x512", kind="column", a=16, cx=32, cy=4, cz=4, tau=0.8, period=200, steps=64,
             k=10, storage="f16", read="planes"),
        # the large column of the benchmark, large spheres
        dict(name="column_128x128x1024", kind="column", a=32, cx=32, cy=4, cz=4, tau=0.6, period=400, steps=32,
             k=10, storage="f32", read="planes"),
        # the source sweep: independent columns of several lengths and sources
        # advanced in one call
        dict(name="sweep_12", kind="sweep", n=12, steps=96, k=2),
        # gradients of the probe misfit of a fixed packing, from rest
        dict(name="adjoint_64x64x512", kind="adjoint", a=32, cx=16, cy=2, cz=2, tau=0.6, steps=200, every=100,
             probe=64),
        # and of the smooth coupling surrogate, sphere positions among them
        dict(name="surrogate_64x64x256", kind="surrogate", a=32, cx=8, cy=2, cz=2, tau=0.6, steps=100, every=50,
             probe=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["column"] * 5 + ["spheres"] * 2 + ["chain", "settle", "dry", "sweep", "adjoint", "surrogate"])
    if kind == "column":
        a = rng.randint(14, 34)
        cy, cz = rng.choice([(1, 1), (2, 2), (4, 4), (1, 2), (3, 2)])
        cx = _log(rng, 4, max(4, min(40, 4_000_000 // (a ** 3 * cy * cz))))
        return dict(kind=kind, a=a, cx=cx, cy=cy, cz=cz, tau=round(rng.uniform(0.6, 1.1), 3),
                    period=_log(rng, 50, 800), steps=rng.choice([16, 32, 48, 64]), k=rng.choice([1, 2, 4, 10]),
                    storage=rng.choice(["f32", "f32", "bf16", "f16"]), read=rng.choice(["fields", "planes", "probe"]))
    if kind == "spheres":
        R = round(rng.uniform(2.5, 7.0), 3)
        nx, ny, nz = (max(int(2 * R) + 6, _log(rng, 20, 120)) for _ in range(3))
        n = max(1, min(400, int(0.12 * nx * ny * nz / (4.2 * R ** 3))))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, n=rng.randint(1, n), R=R, vel=round(rng.uniform(1e-3, 0.02), 4),
                    steps=rng.randint(20, 60), tau=round(rng.uniform(0.6, 1.2), 3), periodic=rng.random() < 0.3)
    if kind == "chain":
        return dict(kind=kind, n=rng.randint(10, 60), steps=rng.choice([32, 64, 96]), k=rng.choice([1, 4, 10]),
                    mobile=rng.random() < 0.7)
    if kind == "settle":
        return dict(kind=kind, L=_log(rng, 24, 160), R=round(rng.uniform(3.0, 9.0), 3),
                    tau=round(rng.uniform(0.8, 1.8), 3), steps=rng.choice([16, 32, 64]))
    if kind == "dry":
        return dict(kind=kind, a=rng.randint(14, 34), cx=_log(rng, 4, 96), cy=rng.randint(1, 4), cz=rng.randint(2, 4),
                    k=rng.choice([2, 10, 20]), steps=rng.choice([32, 64]))
    if kind == "sweep":
        return dict(kind=kind, n=rng.randint(2, 14), steps=rng.randint(32, 97), k=rng.choice([2, 10]))
    a = rng.choice([16, 20, 24, 32])
    c = rng.choice([(4, 1), (8, 1), (6, 2), (12, 2)])
    return dict(kind=kind, a=a, cx=c[0], cy=c[1], cz=c[1], tau=round(rng.uniform(0.58, 0.9), 3),
                steps=rng.randint(60, 140), every=rng.choice([20, 40, 50]), probe=rng.randint(4, 24))


# ---------------------------------------------------------------- inputs

def _workload(c, seed):
    """The seeded input of a case as a workloads.Workload."""
    rng = np.random.default_rng([seed, 1808])
    kind = c["kind"]
    if kind in ("column", "adjoint", "surrogate", "dry"):
        a, R = float(c["a"]), RATIO * c["a"]
        nx, ny, nz = (c["a"] * c[d] for d in ("cx", "cy", "cz"))
        w = workloads.fcc_column(nx, ny, nz, c.get("tau", 0.8), a, R, jitter=1e-3 * R, seed=seed,
                                 period=c.get("period", 200) * rng.uniform(0.95, 1.05), substeps=c.get("k", 1))
        if kind in ("adjoint", "surrogate"):
            w.fixed = np.ones(len(w.R), np.uint8)
            w.omega = 2 * math.pi / 60
            w.probe_x = c["probe"]
        if c.get("read") == "probe":
            w.probe_x = nx // 2
        return w
    if kind == "chain":
        w = workloads.saturated_chain(c["mobile"], n=c["n"], dem_substeps=c["k"])
        w.omega *= rng.uniform(0.9, 1.1)
        w.X[:, 1:] += rng.uniform(-0.2, 0.2, 2)
        w.t_n = -1
        return w
    if kind == "settle":
        L = c["L"]
        return workloads.Workload(name="settle", nx=L, ny=L, nz=L, tau=c["tau"], inlet=workloads.X_PERIODIC,
                                  X=L / 2 + rng.uniform(0, 1, (1, 3)), R=np.array([c["R"]]),
                                  fixed=np.zeros(1, np.uint8), body_force=(0.0, 0.0, 0.1), amplitude=0.0,
                                  dem_substeps=1, mu=0.0)
    w = workloads.random_small(seed, nx=c["nx"], ny=c["ny"], nz=c["nz"], n=c["n"], R=c["R"], tau=c["tau"],
                               vel=c["vel"])
    if c["periodic"]:
        w.inlet = workloads.X_PERIODIC
    w.amplitude, w.omega = 2e-3, 2 * math.pi / 60
    return w


def _sweep(c, seed):
    """The columns of a source sweep: lengths, periods and waveforms as in
    workloads.config_sweep, shorter columns."""
    rng = np.random.default_rng([seed, 44])
    ws = []
    for k in range(c["n"]):
        period = float(np.geomspace(50, 800, c["n"])[k]) * rng.uniform(0.95, 1.05)
        w = workloads.fcc_column(16 * (16 + (k * 11) % 33), 32, 32, 0.8, 16.0, 5.7, jitter=0.01,
                                 seed=int(rng.integers(1 << 30)), period=period, substeps=c["k"])
        if k % 6 == 5:
            w.waveform, w.t0 = workloads.RICKER, period
        ws.append(w)
    return ws


def _target(c, seed, rho_f=1.0):
    """A recorded probe trace to fit: a delayed wave with seeded noise."""
    rng = np.random.default_rng([seed, 7])
    k = np.arange(c["steps"])
    arrive = c["probe"] * math.sqrt(3.0)
    wave = 5e-4 * np.sin(2 * math.pi / 60 * (k - arrive)) * (k > arrive)
    return (rho_f + wave + rng.normal(0.0, 1e-5, c["steps"])) / 3.0


def prepare(c, seed):
    kind = c["kind"]
    if kind == "sweep":
        sims = [lbmdem.Sim.from_workload(w, skin=0.25, dem_skin=0.5) for w in _sweep(c, seed)]
        return dict(case=c, sims=sims, batch=lbmdem.Batch(sims))
    w = _workload(c, seed)
    over = {}
    if kind == "column":
        # the benchmark's re-layout skin; totals recorded where the probe is
        over = dict(storage=STORAGE[c["storage"]], skin=0.1, dem_skin=0.5,
                    monitor_every=16 if c["read"] == "probe" else 0)
    elif kind == "settle":
        over = dict(skin=2.0, dem_skin=2.0)
    elif kind == "dry":
        over = dict(lbm_on=0)
    sim = lbmdem.Sim.from_workload(w, **over)
    return dict(case=c, sim=sim, w=w, target=_target(c, seed) if kind in ("adjoint", "surrogate") else None)


# ---------------------------------------------------------------- one pass

def _f32(a):
    return np.asarray(a, np.float32)


def _scale(storage):
    return 4096.0 if storage == "f16" else 1.0


def _stored(a, storage):
    """An output of the fluid in the form of its storage."""
    if storage == "f32":
        return _f32(a)
    return torch.from_numpy(_f32(_scale(storage) * a)).to(torch.float16 if storage == "f16" else torch.bfloat16)


def _spheres(p, storage="f32"):
    out = {k: p[k] if k == "X" else _f32(p[k]) for k in ("X", "V", "W", "q")}
    return dict(out, Fh=_stored(p["Fh"], storage), Th=_stored(p["Th"], storage))


def _fluid(rho, storage, solid=None):
    """The density, as a deviation from rest where the storage has 16 bits."""
    return rho if storage == "f32" else rho - (1.0 if solid is None else 1.0 * (solid == 0))


def _joined(columns):
    """The columns' outputs one after another, name by name."""
    return {k: np.concatenate([c[k] for c in columns]) for k in columns[0]}


def run(s):
    c, kind = s["case"], s["case"]["kind"]
    if kind == "sweep":
        s["batch"].step(c["steps"])
        s["batch"].sync()
        return _joined([dict(_spheres(g.particles()), rho=_f32(r), jx=_f32(j))
                        for g in s["sims"] for r, j in [g.plane_means()]])
    sim, w = s["sim"], s["w"]
    if kind == "adjoint":
        sim.set_packing(w.X, w.R, None, None, w.fixed)
        loss, d_tau, d_amp, trace = sim.adjoint(c["steps"], c["every"], s["target"])
        return dict(loss=loss, d_tau=d_tau, d_amp=d_amp, trace=_f32(trace))
    if kind == "surrogate":
        loss, d_tau, d_amp, d_x, trace = sim.adjoint_psm(c["steps"], c["every"], s["target"])
        return dict(loss=loss, d_tau=d_tau, d_amp=d_amp, d_x=_f32(d_x), trace=_f32(trace))
    if kind == "spheres":
        sim.set_packing(w.X, w.R, w.V, w.W, w.fixed)
    sim.step(c["steps"])
    st = c.get("storage", "f32")
    out = _spheres(sim.particles(), st)
    if kind == "dry":
        return out
    if kind in ("chain", "spheres") or c.get("read") == "fields":
        rho, u, solid = sim.fields()
        return dict(out, rho=_stored(_fluid(rho, st, solid), st), u=_stored(u, st), solid=solid)
    rho, jx = sim.plane_means()
    out.update(rho=_stored(_fluid(rho, st), st), jx=_stored(jx, st))
    if c.get("read") == "probe":
        out.update(trace=_stored(_fluid(sim.probe(), st), st), totals=_f32(sim.monitors()[:1]))
    return out


# ---------------------------------------------------------------- work

def _updates(c):
    """(fluid-node updates, sphere substeps, bytes per population) of a pass;
    touching spheres' lenses are left out of the solid volume."""
    kind = c["kind"]
    ball = 4.0 / 3.0 * math.pi
    if kind == "sweep":
        cells = sum(16 + (k * 11) % 33 for k in range(c["n"]))
        return c["steps"] * cells * (16 * 32 * 32 - 16 * ball * 5.7 ** 3), c["steps"] * cells * 16 * c["k"], 4
    if kind == "chain":
        return c["steps"] * (620 * 144 - c["n"] * ball * 5.005 ** 3), c["steps"] * c["n"] * c["k"], 4
    if kind == "settle":
        return c["steps"] * (c["L"] ** 3 - ball * c["R"] ** 3), c["steps"], 4
    if kind == "spheres":
        return (c["steps"] * (c["nx"] * c["ny"] * c["nz"] - c["n"] * ball * c["R"] ** 3),
                c["steps"] * c["n"] * 4, 4)
    cells = c["cx"] * c["cy"] * c["cz"]
    fluid = 0 if kind == "dry" else cells * c["a"] ** 3 * (1.0 - 4 * ball * RATIO ** 3)
    if kind == "surrogate":
        fluid = cells * c["a"] ** 3  # every node carries populations
    return c["steps"] * fluid, c["steps"] * 4 * cells * c.get("k", 1), 4 if c.get("storage", "f32") == "f32" else 2


def work(c):
    nodes, substeps, esz = _updates(c)
    # 19 populations read and written per node and step; the gradients read
    # the adjoint and the forward state and write the adjoint besides
    reads = {"adjoint": 5, "surrogate": 5}.get(c["kind"], 2)
    # a sphere's state (about 150 B) once per substep, 12 contacts shared by two spheres
    return {"bytes": nodes * 19 * esz * reads + substeps * 150,
            "flops": nodes * 250 * (reads / 2) + substeps * 6 * 150}


# ---------------------------------------------------------------- FP64

# D3Q19 in the library's documented order (the columns of Eq. 3)
_C = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (1, -1, 0), (1, 0, 1),
      (1, 0, -1), (-1, 1, 0), (-1, -1, 0), (-1, 0, 1), (-1, 0, -1), (0, 1, 1), (0, 1, -1), (0, -1, 1), (0, -1, -1),
      (0, 0, 0)]
_W = [1 / 3 if not any(v) else 1 / 18 if sum(map(abs, v)) == 1 else 1 / 36 for v in _C]
_OPP = [_C.index(tuple(-x for x in v)) for v in _C]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _cross(a, b):
    return torch.linalg.cross(a, b)


def _collide(g, om, rho_f):
    """Eqs. 4, 6, 7 on the deviations g[19] = f - w rho_f; (1 - om) g + om g^eq."""
    d = sum(g)
    j = [sum(v[a] * x for v, x in zip(_C, g) if v[a]) for a in range(3)]
    rho = rho_f + d
    u = [x / rho for x in j]
    uu = 1.5 * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2])
    eq = []
    for v, wt in zip(_C, _W):
        cu = v[0] * u[0] + v[1] * u[1] + v[2] * u[2]
        eq.append(wt * (d + rho * (3 * cu + 4.5 * cu * cu - uu)))
    return d, u, eq, [(1 - om) * x + om * e for x, e in zip(g, eq)]


def _face(f, drho, sgn):
    """Section 2.4 on the 19 deviations f of an x face's nodes; sgn = +1 at the inlet."""
    rest = f[18] + f[2] + f[3] + f[4] + f[5] + f[14] + f[15] + f[16] + f[17]
    ny = 0.5 * (f[2] + f[14] + f[15] - f[3] - f[16] - f[17])
    nz = 0.5 * (f[4] + f[14] + f[16] - f[5] - f[15] - f[17])
    f = list(f)
    if sgn > 0:
        j = drho - (rest + 2 * (f[1] + f[10] + f[11] + f[12] + f[13]))
        f[0], f[6], f[7] = f[1] + j / 3, f[11] + j / 6 - ny, f[10] + j / 6 + ny
        f[8], f[9] = f[13] + j / 6 - nz, f[12] + j / 6 + nz
    else:
        j = rest + 2 * (f[0] + f[6] + f[7] + f[8] + f[9]) - drho
        f[1], f[11], f[10] = f[0] - j / 3, f[6] - j / 6 + ny, f[7] - j / 6 - ny
        f[13], f[12] = f[8] - j / 6 + nz, f[9] - j / 6 - nz
    return f


def _shape(w, t):
    """Eq. 25 / Table 2: the source per unit amplitude at time t."""
    if 0 <= w.t_n < t:
        return 0.0
    if w.waveform == workloads.RICKER:
        a = 0.5 * w.omega * (t - w.t0)
        return (1 - 2 * a * a) * math.exp(-a * a)
    return math.sin(w.omega * t)


def _ends(w, fn, amp, t, fluid_up):
    """Inlet and outlet of the streamed state fn (Section 2.4)."""
    if w.inlet == workloads.X_PERIODIC:
        return fn
    first = [x[:1] for x in fn]
    if w.inlet == workloads.INLET_PRESSURE:
        first = _face(first, amp * _shape(w, t), +1)
    last = [x[-1:] for x in fn]
    if w.outlet == workloads.OUTLET_PRESSURE:
        last = _face(last, 0.0, -1)
    elif w.outlet == workloads.OUTLET_ZERO_GRADIENT:
        last = [torch.where(fluid_up, y[-2:-1], x) if v[0] < 0 else x for v, x, y in zip(_C, last, fn)]
    return [torch.cat([a, x[1:-1], b]) for a, x, b in zip(first, fn, last)]


class _Exact:
    """The coupled step in FP64: dense two-lattice streaming, every sphere
    painted anew each step, all contacts from a pair list."""

    def __init__(self, w, lbm=True):
        self.w, self.dev, self.lbm = w, _device(), lbm
        d = dict(device=self.dev, dtype=torch.float64)
        self.X = torch.tensor(np.asarray(w.X), **d).reshape(-1, 3)
        n = self.n = self.X.shape[0]
        self.R = torch.tensor(np.asarray(w.R), **d)
        z = torch.zeros(n, 3, **d)
        self.V = z.clone() if w.V is None else torch.tensor(w.V, **d)
        self.W = z.clone() if w.W is None else torch.tensor(w.W, **d)
        self.q = torch.zeros(n, 4, **d)
        self.q[:, 0] = 1
        self.free = torch.tensor(np.asarray(w.fixed) == 0, device=self.dev)[:, None]
        self.V, self.W = self.V * self.free, self.W * self.free
        self.m = (w.rho_p * 4 / 3 * math.pi * self.R ** 3)[:, None]
        self.I = 0.4 * self.m * self.R[:, None] ** 2
        self.Fh, self.Th, self.Fp, self.Tp = z.clone(), z.clone(), z.clone(), z.clone()
        self.t, self.trace = 0, []
        self.px = w.inlet == workloads.X_PERIODIC
        self.L = torch.tensor([w.nx, w.ny, w.nz], **d)
        self.per = torch.tensor([self.px, True, True], device=self.dev)
        self.shape = (w.nx, w.ny, w.nz)
        self.N = w.nx * w.ny * w.nz
        self._pairs()
        self.Fc, self.Tc = self._contacts(self.V, self.W, 0.0)
        if lbm:
            self.own = self._paint()
            self._links()
            self.g = [torch.zeros(self.shape, **d) for _ in range(19)]

    # ---- spheres (Eqs. 9-12)
    def _pairs(self):
        """Pairs i < j with the periodic image of j, wide enough for the pass."""
        w, n = self.w, self.n
        reach = 0.0 if w.V is None else 2.0
        out = []
        k = [-1, 0, 1]
        for i0 in range(0, n, 512):
            i = torch.arange(i0, min(n, i0 + 512), device=self.dev)
            d0 = self.X[None] - self.X[i][:, None]
            up = torch.arange(n, device=self.dev)[None] > i[:, None]
            base = -torch.round(d0 / self.L) * self.per
            for kx in k if self.px else [0]:
                for ky in k:
                    for kz in k:
                        s = base + torch.tensor([kx, ky, kz], device=self.dev)
                        dd = ((d0 + s * self.L) ** 2).sum(-1).sqrt()
                        ok = up & (dd < self.R[None] + self.R[i][:, None] + 0.5 + reach)
                        a, b = ok.nonzero(as_tuple=True)
                        out.append((i[a], b, s[a, b] * self.L))
        self.pi, self.pj, self.ps = (torch.cat(x) for x in zip(*out)) if out else (None, None, None)
        self.ft = torch.zeros(0 if self.pi is None else len(self.pi), 3, device=self.dev, dtype=torch.float64)

    def _contacts(self, V, W, dt):
        F, T = torch.zeros_like(self.X), torch.zeros_like(self.X)
        if self.pi is None or not len(self.pi):
            return F, T
        w, i, j = self.w, self.pi, self.pj
        d = self.X[j] + self.ps - self.X[i]
        dist = d.norm(dim=1, keepdim=True)
        Ri, Rj = self.R[i][:, None], self.R[j][:, None]
        delta = (Ri + Rj - dist).clamp(min=0)
        n = d / dist
        sq = (Ri * Rj / (Ri + Rj) * delta).sqrt()
        fn = 2 * w.E_p / (3 * (1 - w.nu_p ** 2)) * sq * delta
        ri, rj = (Ri - delta / 2) * n, -(Rj - delta / 2) * n
        vr = V[j] + _cross(W[j], rj) - V[i] - _cross(W[i], ri)
        vt = vr - (vr * n).sum(1, keepdim=True) * n
        ft = self.ft - (self.ft * n).sum(1, keepdim=True) * n + 2 * w.E_p / (
            (1 + w.nu_p) * (2 - w.nu_p)) * sq * dt * vt
        m = ft.norm(dim=1, keepdim=True)
        ft = ft * torch.where(m > w.mu * fn, w.mu * fn / m.clamp(min=1e-300), torch.ones_like(m))
        self.ft = ft * (delta > 0)
        f = (-fn * n + self.ft) * (delta > 0)
        F.index_add_(0, i, f).index_add_(0, j, -f)
        T.index_add_(0, i, _cross(ri, f)).index_add_(0, j, _cross(rj, -f))
        return F, T

    def _dem(self):
        w = self.w
        Fa, Ta = 0.5 * (self.Fh + self.Fp), 0.5 * (self.Th + self.Tp)
        self.Fp, self.Tp = self.Fh, self.Th
        Fa = Fa + torch.tensor(w.body_force, device=self.dev, dtype=torch.float64)
        dt = 1.0 / w.dem_substeps
        for _ in range(w.dem_substeps):
            vh = (self.V + 0.5 * dt * (self.Fc + Fa) / self.m) * self.free
            wh = (self.W + 0.5 * dt * (self.Tc + Ta) / self.I) * self.free
            self.X = self.X + dt * vh
            q0, qv = self.q[:, :1], self.q[:, 1:]
            q = self.q + 0.5 * dt * torch.cat([-(wh * qv).sum(1, keepdim=True), q0 * wh + _cross(wh, qv)], 1)
            self.q = torch.where(self.free, q / q.norm(dim=1, keepdim=True), self.q)
            self.Fc, self.Tc = self._contacts(vh, wh, dt)
            self.V = (vh + 0.5 * dt * (self.Fc + Fa) / self.m) * self.free
            self.W = (wh + 0.5 * dt * (self.Tc + Ta) / self.I) * self.free

    # ---- solid map (Section 2.3)
    def _paint(self):
        own = torch.full((self.N,), 1 << 30, device=self.dev, dtype=torch.int64)
        if self.n:
            r = int(math.ceil(float(self.R.max()))) + 1
            o = torch.arange(-r, r + 1, device=self.dev)
            box = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
            best = torch.full((self.N,), math.inf, device=self.dev, dtype=torch.float64)
            hits = []
            L = torch.tensor(self.shape, device=self.dev)
            for p0 in range(0, self.n, 256):
                X = self.X[p0:p0 + 256]
                node = torch.floor(X).long()[:, None] + box
                d2 = ((node - X[:, None]) ** 2).sum(-1)
                R2 = self.R[p0:p0 + 256, None] ** 2
                ok = d2 < R2
                if not self.px:
                    ok &= (node[..., 0] > 0) & (node[..., 0] < self.shape[0] - 1)
                p, k = ok.nonzero(as_tuple=True)
                nd = node[p, k] % L
                flat = (nd[:, 0] * self.shape[1] + nd[:, 1]) * self.shape[2] + nd[:, 2]
                ratio = (d2 / R2)[p, k]
                best.scatter_reduce_(0, flat, ratio, "amin")
                hits.append((flat, ratio, p + p0))
            for flat, ratio, p in hits:
                win = ratio == best[flat]
                own.scatter_reduce_(0, flat[win], p[win], "amin")
        own[own == 1 << 30] = -1
        return own

    def _xyz(self, flat):
        _, ny, nz = self.shape
        return torch.stack([flat // (ny * nz), flat // nz % ny, flat % nz], 1).double()

    def _lever(self, pos, p):
        d = pos - self.X[p]
        return d - self.per * self.L * torch.floor(d / self.L + 0.5)

    def _links(self):
        """Per direction m: the fluid nodes whose upstream neighbour (x - c_m)
        is solid, and where the population comes back from an x end."""
        o = self.own.reshape(self.shape)
        fl = o < 0
        self.lk = []
        for v in _C[:18]:
            up = torch.roll(o, v, (0, 1, 2))
            end = torch.zeros(self.shape, device=self.dev, dtype=torch.bool)
            if not self.px and v[0]:
                end[0 if v[0] > 0 else -1] = True
            hit = (fl & (up >= 0) & ~end).reshape(-1).nonzero()[:, 0]
            self.lk.append((hit, up.reshape(-1)[hit], end))

    def _convert(self):
        """Eqs. 16-17 with the newly painted map."""
        new = self._paint()
        old, w = self.own, self.w
        cov = ((old < 0) & (new >= 0)).nonzero()[:, 0]
        unc = ((old >= 0) & (new < 0)).nonzero()[:, 0]
        if len(cov):
            p = new[cov]
            f = torch.stack([x.reshape(-1)[cov] for x in self.g])
            j = torch.stack([sum(v[a] * x for v, x in zip(_C, f) if v[a]) for a in range(3)], 1)
            self.Fh.index_add_(0, p, j)
            self.Th.index_add_(0, p, _cross(self._lever(self._xyz(cov), p), j))
        if len(unc):
            p, pos = old[unc], self._xyz(unc)
            tot, cnt = torch.zeros(len(unc), **self._d()), torch.zeros(len(unc), **self._d())
            L = torch.tensor(self.shape, device=self.dev)
            for v in _C[:18]:
                nb = pos.long() + torch.tensor(v, device=self.dev)
                ok = torch.ones(len(unc), device=self.dev, dtype=torch.bool)
                if not self.px:
                    ok = (nb[:, 0] >= 0) & (nb[:, 0] < L[0])
                nb = nb % L
                k = (nb[:, 0] * L[1] + nb[:, 1]) * L[2] + nb[:, 2]
                ok = ok & (old[k] < 0)
                tot += torch.where(ok, w.rho_f + sum(x.reshape(-1)[k] for x in self.g), 0.0)
                cnt += ok
            rb = torch.where(cnt > 0, tot / cnt.clamp(min=1), w.rho_f)
            r = self._lever(pos, p)
            vb = self.V[p] + _cross(self.W[p], r)
            uu = 1.5 * (vb * vb).sum(1)
            for m, v in enumerate(_C):
                cu = vb @ torch.tensor(v, **self._d())
                self.g[m].reshape(-1)[unc] = _W[m] * (rb - w.rho_f + rb * (3 * cu + 4.5 * cu * cu - uu))
            self.Fh.index_add_(0, p, -rb[:, None] * vb)
            self.Th.index_add_(0, p, -_cross(r, rb[:, None] * vb))
        if not torch.equal(old, new):  # nodes may also pass from sphere to sphere
            self.own = new
            self._links()

    def _d(self):
        return dict(device=self.dev, dtype=torch.float64)

    def _fluid(self):
        w = self.w
        self._convert()
        fl = self.own.reshape(self.shape) < 0
        if w.probe_x >= 0:
            m = fl[w.probe_x]
            self.trace.append(float(w.rho_f + sum(x[w.probe_x] for x in self.g)[m].mean()))
        g = [torch.where(fl, x, 0.0) for x in self.g]
        _, _, _, post = _collide(g, 1 / w.tau, w.rho_f)
        del g
        fn = []
        for m, v in enumerate(_C):
            if m == 18:
                fn.append(post[18])
                continue
            hit, p, end = self.lk[m]
            x = torch.where(end, post[_OPP[m]], torch.roll(post[m], v, (0, 1, 2)))
            if len(hit):
                c = -torch.tensor(v, **self._d())  # from the node towards the wall
                r = self._lever(self._xyz(hit) + 0.5 * c, p)
                cv = (self.V[p] + _cross(self.W[p], r)) @ c
                out = post[_OPP[m]].reshape(-1)[hit]
                back = out - 6 * _W[m] * w.rho_f * cv
                x.reshape(-1)[hit] = back
                f = (out + back)[:, None] * c
                self.Fh.index_add_(0, p, f)
                self.Th.index_add_(0, p, _cross(r, f))
            fn.append(x)
        self.g = _ends(w, fn, w.amplitude, self.t + 1, fl[-2:-1])

    def step(self, n):
        for _ in range(n):
            self.Fh, self.Th = torch.zeros_like(self.X), torch.zeros_like(self.X)
            if self.lbm:
                self._fluid()
            if self.n:
                self._dem()
            self.t += 1

    # ---- read-outs, as the library lays them out
    def spheres(self):
        p = dict(X=self.X, V=self.V, W=self.W, q=self.q, Fh=self.Fh, Th=self.Th)
        return {k: x.cpu().numpy() for k, x in p.items()}

    def _moments(self):
        fl = self.own.reshape(self.shape) < 0
        d = sum(self.g)
        j = [sum(v[a] * x for v, x in zip(_C, self.g) if v[a]) for a in range(3)]
        return fl, d, j

    def fields(self):
        fl, d, j = self._moments()
        rho = torch.where(fl, self.w.rho_f + d, 0.0)
        u = torch.stack([torch.where(fl, x / (self.w.rho_f + d), 0.0) for x in j])
        return rho.cpu().numpy(), u.cpu().numpy(), (~fl).cpu().numpy()

    def planes(self):
        fl, d, j = self._moments()
        n = fl.sum((1, 2))
        mean = lambda x: (torch.where(fl, x, 0.0).sum((1, 2)) / n).cpu().numpy()  # noqa: E731
        return self.w.rho_f + mean(d), mean(j[0])


def _fixed_gradient(c, seed):
    """The probe misfit of a fixed packing and its gradient by autograd."""
    w = _workload(c, seed)
    e = _Exact(w)
    dev, fl = e.dev, e.own.reshape(e.shape) < 0
    back = []
    for m, v in enumerate(_C[:18]):
        hit, _, end = e.lk[m]
        b = end.clone()
        b.view(-1)[hit] = True
        back.append(b)
    tau = torch.tensor(w.tau, device=dev, dtype=torch.float64, requires_grad=True)
    amp = torch.tensor(w.amplitude, device=dev, dtype=torch.float64, requires_grad=True)
    probe = fl[w.probe_x]

    def step(g, tau, amp, t):
        _, _, _, post = _collide([x * fl for x in g.unbind(0)], 1 / tau, w.rho_f)
        fn = [torch.where(back[m], post[_OPP[m]], torch.roll(post[m], v, (0, 1, 2))) if m < 18 else post[18]
              for m, v in enumerate(_C)]
        return torch.stack(_ends(w, fn, amp, t, fl[-2:-1]))

    loss, trace = _rollout(c, seed, step, torch.stack(e.g), tau, amp,
                           lambda g: w.rho_f + g[:, w.probe_x].sum(0)[probe].mean())
    return dict(loss=loss, d_tau=float(tau.grad), d_amp=float(amp.grad), trace=trace)


def _rollout(c, seed, step, g, tau, amp, probe):
    """Loss and trace over the case's steps, one state kept per step."""
    target = torch.tensor(_target(c, seed), device=g.device, dtype=torch.float64)
    states, press = [g], []
    with torch.no_grad():
        for t in range(c["steps"]):
            press.append(float(probe(states[-1])) / 3)
            states.append(step(states[-1], tau, amp, t + 1))
    press = np.array(press)
    loss = float(((press - target.cpu().numpy()) ** 2).sum())
    lam = torch.zeros_like(g)
    for t in reversed(range(c["steps"])):
        s = states[t].detach().requires_grad_(True)
        states[t + 1] = None
        out = (step(s, tau, amp, t + 1) * lam).sum() + (probe(s) / 3 - target[t]) ** 2
        out.backward()
        lam = s.grad
    return loss, press


def _surrogate_gradient(c, seed):
    """The coupling surrogate (solid-fraction-weighted collision) and its
    gradient by autograd, sphere positions included."""
    w = _workload(c, seed)
    dev = _device()
    d = dict(device=dev, dtype=torch.float64)
    shape = (w.nx, w.ny, w.nz)
    X = torch.tensor(w.X, **d)
    R, L = float(w.R[0]), torch.tensor([w.ny, w.nz], device=dev)
    r = int(math.ceil(R)) + 2
    o = torch.arange(-r, r + 1, device=dev)
    box = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
    node = torch.floor(X).long()[:, None] + box
    off = node - X[:, None]
    dist = off.norm(dim=-1)
    v = (R - dist + 0.5).clamp(0, 1)
    ok = (v > 0) & (node[..., 0] > 0) & (node[..., 0] < w.nx - 1)
    yz = node[..., 1:] % L
    flat = ((node[..., 0] * w.ny + yz[..., 0]) * w.nz + yz[..., 1])[ok]
    ep = (v * v * (3 - 2 * v))[ok]
    keep = torch.ones(w.nx * w.ny * w.nz, **d).scatter_reduce_(0, flat, 1 - ep, "prod")
    eps = (1 - keep).reshape(shape).requires_grad_(True)
    tau = torch.tensor(w.tau, **d, requires_grad=True)
    amp = torch.tensor(w.amplitude, **d, requires_grad=True)
    up = torch.ones(1, w.ny, w.nz, device=dev, dtype=torch.bool)

    def step(g, tau, amp, t):
        g = g.unbind(0)
        rho, _, eq, _ = _collide(g, 1 / tau, w.rho_f)
        B = eps * (tau - 0.5) / ((1 - eps) + (tau - 0.5))
        post = [g[m] - (1 - B) / tau * (g[m] - eq[m]) + B * (g[_OPP[m]] - g[m] + _W[m] * rho - eq[_OPP[m]])
                for m in range(19)]
        fn = []
        for m, v in enumerate(_C):
            x = torch.roll(post[m], v, (0, 1, 2))
            if v[0] > 0:
                x = torch.cat([post[_OPP[m]][:1], x[1:]])
            elif v[0] < 0:
                x = torch.cat([x[:-1], post[_OPP[m]][-1:]])
            fn.append(x)
        return torch.stack(_ends(w, fn, amp, t, up))

    loss, trace = _rollout(c, seed, step, torch.zeros(19, *shape, **d), tau, amp,
                           lambda g: w.rho_f + g[:, w.probe_x].sum(0).mean())
    G = eps.grad.reshape(-1)[flat]
    slope = (6 * v * (1 - v))[ok]
    f = torch.where(slope > 0, G * keep[flat] / (1 - ep).clamp(min=1e-300) * slope / dist[ok].clamp(min=1e-300), 0.0)
    dX = torch.zeros_like(X).index_add_(0, ok.nonzero()[:, 0], f[:, None] * off[ok])
    return dict(loss=loss, d_tau=float(tau.grad), d_amp=float(amp.grad), d_x=dX.cpu().numpy(), trace=trace)


def exact(c, seed):
    kind = c["kind"]
    if kind == "adjoint":
        return _fixed_gradient(c, seed)
    if kind == "surrogate":
        return _surrogate_gradient(c, seed)
    if kind == "sweep":
        out = []
        for w in _sweep(c, seed):
            e = _Exact(w)
            e.step(c["steps"])
            rho, jx = e.planes()
            out.append(dict(e.spheres(), rho=rho, jx=jx))
        return _joined(out)
    w = _workload(c, seed)
    e = _Exact(w, lbm=kind != "dry")
    e.step(c["steps"])
    st = c.get("storage", "f32")
    sc = _scale(st)
    out = e.spheres()
    out.update(Fh=sc * out["Fh"], Th=sc * out["Th"])
    if kind == "dry":
        return out
    if kind in ("chain", "spheres") or c.get("read") == "fields":
        rho, u, solid = e.fields()
        return dict(out, rho=sc * _fluid(rho, st, solid), u=sc * u, solid=None)
    rho, jx = e.planes()
    out.update(rho=sc * _fluid(rho, st), jx=sc * jx)
    if c.get("read") == "probe":
        out.update(trace=sc * _fluid(np.array(e.trace), st), totals=None)
    return out
