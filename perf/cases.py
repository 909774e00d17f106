"""Workloads of the lattice update as a user's program runs them, for timing and for comparison.

A pass advances a lattice (or an ensemble) by some time steps through the public binding and reads
the macroscopic fields of the new state, the way a simulation loop does between two outputs.  The
cases cover the geometries that the package's workloads describe (static and evaporating droplets,
pool boiling, nucleate boiling on a wetting wall, a sessile drop), a closed box with solid walls on
every face, each storage type, both temperature lattices and the batched ensemble; sizes are those of
the benchmark, the parity tests and the storage studies, or generic.

`exact` restates one run in FP64 with plain torch operations.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2201_06039_gb300 import lbm

PERIODIC, WALL, OUTFLOW, THERMAL = 0, 1, 2, 3
B_EOS, R_EOS, ACENTRIC = 2.0 / 21.0, 1.0, 0.344
PRECISION = {"fp32": 0, "bf16": 1, "fp16": 2}

# coexistence densities (liquid, vapour) of the Peng-Robinson EOS at T / Tc (equal areas); in these
# units they do not depend on the constant a
COEXIST = {0.80: (7.20385, 0.197122), 0.82: (6.98797, 0.246548), 0.84: (6.75401, 0.306578),
           0.86: (6.49895, 0.379679), 0.88: (6.21877, 0.469233), 0.90: (5.90790, 0.580099)}

# Per kind: faces (-x, +x, -y, +y, -z, +z), face temperatures over Tc, EOS constant a, the matching
# sigma of the forcing term, and the other parameters that differ from the library's defaults.
KINDS = {
    # a liquid drop at rest in its vapour, periodic box: the parity and spurious-current run (only run
    # for some steps from fresh fields: the small periodic drops diverge after 10^4 steps)
    "droplet": dict(bc=(PERIODIC,) * 6, Tw=(0.86,) * 6, a=2 / 49, sigma=0.1125),
    # a drop that evaporates into hotter vapour held by the faces, constant conductivity
    "evaporation": dict(bc=(THERMAL,) * 6, Tw=(0.95,) * 6, a=1 / 49, sigma=0.1175, lambda_mode=1, chi=0.2),
    # a liquid pool over a wall with a hot spot, open top: the benchmark's workload
    "pool": dict(bc=(PERIODIC,) * 4 + (WALL, OUTFLOW), Tw=(0.86,) * 6, a=2 / 49, sigma=0.1125, hot=0.10,
                 gz=-3e-5, rho_buoy=0.37968),
    # nucleate boiling: hot bottom wall with a hydrophobic square in a hydrophilic rest, closed top
    "nucleate": dict(bc=(PERIODIC,) * 4 + (WALL, WALL), Tw=(0.86, 0.86, 0.86, 0.86, 0.96, 0.86), a=2 / 49,
                     sigma=0.1125, gz=-1.5e-5, wet=(1.40, 0.0, 1.0, 0.284)),
    # a sessile drop settling on a neutral wall with the temperature frozen, before evaporation starts
    "sessile": dict(bc=(PERIODIC,) * 4 + (WALL, WALL), Tw=(0.86, 0.86, 0.86, 0.86, 0.87, 0.86), a=1 / 49,
                    sigma=0.1175, chi=0.02, wet=(1.0, 0.005, 1.0, 0.005), thermal_off=1),
    # a closed box half full of liquid, solid walls on all six faces, bottom a little warmer
    "cavity": dict(bc=(WALL,) * 6, Tw=(0.86, 0.86, 0.86, 0.86, 0.88, 0.86), a=2 / 49, sigma=0.1125, gz=-3e-5),
}


def listed():
    return [
        # smallest call: a parity-test sized drop, library defaults throughout (the state is checked in
        # every lbm_step)
        dict(name="evaporation_32", kind="evaporation", nx=32, ny=32, nz=32, steps=50, check=True),
        # D^2-law run, thermal-only faces and constant conductivity
        dict(name="evaporation_128", kind="evaporation", nx=128, ny=128, nz=128, steps=10),
        # the benchmark lattice, FP32 storage
        dict(name="pool_200x200x300", kind="pool", nx=200, ny=200, nz=300, steps=10),
        # the same in shifted BF16 storage (the benchmark reports it beside FP32)
        dict(name="pool_200x200x300_bf16", kind="pool", nx=200, ny=200, nz=300, steps=10, precision="bf16"),
        # the downscaled pool of the storage-error study, shifted FP16 storage
        dict(name="pool_64x64x96_fp16", kind="pool", nx=64, ny=64, nz=96, steps=20, precision="fp16"),
        # bubble nucleation and departure on a wetting wall with a patch
        dict(name="nucleate_200x200x280", kind="nucleate", nx=200, ny=200, nz=280, steps=10),
        # settling stage of the heated-surface droplet (isothermal: g frozen)
        dict(name="sessile_200x200x100", kind="sessile", nx=200, ny=200, nz=100, steps=10),
        # solid walls on every face, no extent a multiple of a tile
        dict(name="cavity_150x110x130", kind="cavity", nx=150, ny=110, nz=130, steps=10),
        # the evaporating droplet on the D3Q19 temperature lattice
        dict(name="evaporation_128_q19", kind="evaporation", nx=128, ny=128, nz=128, steps=5, thermal_q=19),
        # the finite-difference div u option on the downscaled pool (two-pass kernels)
        dict(name="pool_64x64x96_fd_divu", kind="pool", nx=64, ny=64, nz=96, steps=20, divu_mode=1),
        # ensemble of 256 uneven droplets and slabs, autotuned as the benchmark does
        dict(name="ensemble_256", kind="ensemble", count=256, lo=24, hi=96, steps=5),
        # one run of a parameter sweep: host fields in, 20 steps, host fields and totals out, in a
        # context that the sweep keeps
        dict(name="sweep_job_96x80x112", kind="droplet", nx=96, ny=80, nz=112, steps=20, job=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["evaporation", "evaporation", "pool", "pool", "nucleate", "sessile", "cavity", "q19", "divu",
                       "ensemble", "job"])
    if kind == "ensemble":
        lo = rng.randint(24, 40)
        return dict(kind="ensemble", count=_log(rng, 4, 192), lo=lo, hi=rng.randint(lo + 8, 96), steps=rng.randint(2, 5))
    if kind in ("evaporation", "job"):
        c = dict(kind="droplet" if kind == "job" else kind, nx=_log(rng, 24, 160), ny=_log(rng, 24, 160),
                 nz=_log(rng, 24, 160), steps=rng.randint(5, 40))
        c.update(dict(job=True) if kind == "job" else dict(check=rng.random() < 0.5))
        return c
    if kind == "q19":
        return dict(kind="evaporation", nx=_log(rng, 32, 144), ny=_log(rng, 32, 128), nz=_log(rng, 32, 128),
                    steps=rng.randint(3, 10), thermal_q=19)
    if kind == "divu":
        return dict(kind="pool", nx=_log(rng, 40, 128), ny=_log(rng, 40, 128), nz=_log(rng, 48, 128),
                    steps=rng.randint(5, 20), divu_mode=1)
    c = dict(kind=kind, nx=_log(rng, 48, 220), ny=_log(rng, 48, 200), nz=_log(rng, 40, 270), steps=rng.randint(4, 10))
    if kind == "pool":
        c["precision"] = rng.choice(["fp32", "bf16", "fp16"])
    return c


# ----------------------------------------------------------------------------- inputs
def _tc(a):
    return 0.0778 * a / (0.45724 * B_EOS * R_EOS)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(seed)


def _tanh(r, R0, W, inside, outside):
    return 0.5 * (inside + outside) - 0.5 * (inside - outside) * torch.tanh(2.0 * (r - R0) / W)


def _grid(nx, ny, nz):
    d = dict(device=_device(), dtype=torch.float32)
    return (torch.arange(nx, **d)[None, None, :], torch.arange(ny, **d)[None, :, None],
            torch.arange(nz, **d)[:, None, None])


def _noisy(rho, gen):
    return (rho + (2e-3 * torch.rand(rho.shape, generator=gen, device=rho.device) - 1e-3)).contiguous()


def _fields(case, seed):
    """Initial (rho, T, u) of a single lattice: float32 tensors, u of a sweep job only."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    K = KINDS[case["kind"]]
    Tc, gen, rng = _tc(K["a"]), _generator(seed), random.Random(seed)
    x, y, z = _grid(nx, ny, nz)
    rl, rv = COEXIST[0.86]
    off = [rng.uniform(-1.0, 1.0) for _ in range(3)]
    T = torch.full((nz, ny, nx), 0.86 * Tc, device=x.device, dtype=torch.float32)
    u = None
    if case["kind"] in ("droplet", "evaporation"):
        r = torch.sqrt((x - nx / 2 - off[0]) ** 2 + (y - ny / 2 - off[1]) ** 2 + (z - nz / 2 - off[2]) ** 2)
        R0 = (0.25 if case["kind"] == "droplet" else 0.1875) * min(nx, ny, nz)
        rho = _tanh(r, R0, 4.0, rl, rv)
        if case["kind"] == "evaporation":
            T = torch.where(r <= R0, 0.86 * Tc, 0.95 * Tc).to(torch.float32)
        if case.get("job"):   # a sweep also sets a velocity: a weak shear wave
            u = torch.zeros((3, nz, ny, nx), device=x.device)
            u[0] = 5e-3 * torch.sin(2 * math.pi * (y / ny + 0.1 * off[0]))
            u[2] = 5e-3 * torch.cos(2 * math.pi * x / nx)
    elif case["kind"] == "sessile":
        r = torch.sqrt((x - nx / 2 - off[0]) ** 2 + (y - ny / 2 - off[1]) ** 2 + (z + 0.5) ** 2)
        rho = _tanh(r, 0.15 * min(nx, ny, 2 * nz), 4.0, rl, 0.42)
    else:
        height = {"pool": 1 / 3, "nucleate": 5 / 7, "cavity": 1 / 2}[case["kind"]] * nz + off[2]
        rho = _tanh(z + 0 * (x + y), height, 4.0, rl, rv)
    return _noisy(rho, gen), T.contiguous(), u


def _instances(case):
    """(edge, T / Tc, radius over edge) of every instance of an ensemble."""
    rng = random.Random(20220116)
    return [(rng.randint(case["lo"], case["hi"]), rng.choice(sorted(COEXIST)), rng.uniform(0.20, 0.35))
            for _ in range(case["count"])]


def _ensemble_fields(case, seed):
    """Per instance (rho, T): droplets and flat slabs in turn, interfaces 6 wide."""
    gen, rng, Tc = _generator(seed), random.Random(seed), _tc(1 / 49)
    out = []
    for i, (n, tr, frac) in enumerate(_instances(case)):
        x, y, z = _grid(n, n, n)
        off = rng.uniform(-1.0, 1.0)
        rl, rv = COEXIST[tr]
        if i % 2 == 0:
            r = torch.sqrt((x - n / 2 - off) ** 2 + (y - n / 2) ** 2 + (z - n / 2) ** 2)
        else:
            r = (z - n / 2 - off).abs() + 0 * (x + y)
        rho = _noisy(_tanh(r, frac * n, 6.0, rl, rv), gen)
        out.append((rho, torch.full_like(rho, tr * Tc)))
    return out


def _params(case, rho_mean=None):
    p = lbm.lbm_params_default()
    kind = "droplet" if case["kind"] == "ensemble" else case["kind"]
    K = dict(KINDS[kind])
    if case["kind"] == "ensemble":   # the ensemble's EOS constant and sigma
        K.update(a=1 / 49, sigma=0.1175)
    else:
        p.nx, p.ny, p.nz = case["nx"], case["ny"], case["nz"]
    p.a, p.b, p.R, p.acentric, p.sigma = K["a"], B_EOS, R_EOS, ACENTRIC, K["sigma"]
    Tc = _tc(K["a"])
    for f in range(6):
        p.bc[f] = K["bc"][f]
        p.T_wall[f] = K["Tw"][f] * Tc
    p.lambda_mode, p.chi_or_lambda = K.get("lambda_mode", 0), K.get("chi", 0.08)
    p.g[2] = K.get("gz", 0.0)
    p.rho_buoy = K.get("rho_buoy", 0.0)
    p.thermal_off = K.get("thermal_off", 0)
    p.divu_mode = case.get("divu_mode", 0)
    p.thermal_q = case.get("thermal_q", 7)
    if "hot" in K:
        p.hot_dT, p.hot_sigma = K["hot"] * Tc, _hot_sigma(case)
    if "wet" in K:
        p.wall_scheme = 1
        p.wall_phi, p.wall_drho, p.wall_phi_patch, p.wall_drho_patch = K["wet"]
        p.wall_patch_half = _patch_half(case)
    if case.get("precision", "fp32") != "fp32":
        p.precision, p.rho_ref, p.T_ref = PRECISION[case["precision"]], rho_mean, 0.86 * Tc
    # long runs check the state now and then (the totals) instead of in every lbm_step, the default
    p.check_nonfinite = 1 if case.get("check") or case.get("job") else 0
    return p


def _hot_sigma(case):
    return 10.0 * min(case["nx"], case["ny"]) / 200.0


def _patch_half(case):
    return 27.5 * min(case["nx"], case["ny"]) / 200.0 if case["kind"] == "nucleate" else 0.0


# ----------------------------------------------------------------------------- one pass
FIELDS = ("rho", "ux", "uy", "uz", "T")


def prepare(case, seed):
    if case["kind"] == "ensemble":
        inst = _ensemble_fields(case, seed)
        rho = torch.cat([r.ravel() for r, _ in inst])
        T = torch.cat([t.ravel() for _, t in inst])
        batch = lbm.Batch(_params(case), [r.shape[::-1] for r, _ in inst])
        batch.init(rho, T)
        batch.step(1)
        batch.autotune(2)
        return dict(case=case, batch=batch, out={k: torch.empty_like(rho) for k in FIELDS})
    rho, T, u = _fields(case, seed)
    mean = float(rho.double().mean()) if case.get("precision", "fp32") != "fp32" else None
    lat = lbm.Lattice(_params(case, mean))
    if case.get("job"):
        host = [f.cpu().pin_memory() for f in (rho, T, u)]
        out = {k: torch.empty(rho.shape, dtype=torch.float32).pin_memory() for k in FIELDS}
        return dict(case=case, lat=lat, host=host, out=out)
    lat.init(rho, T, u)
    return dict(case=case, lat=lat, out={k: torch.empty_like(rho) for k in FIELDS})


def run(state):
    case, out = state["case"], state["out"]
    if "batch" in state:
        state["batch"].step(case["steps"])
        lbm.lbm_batch_get_moments(state["batch"].b, *[out[k] for k in FIELDS])
        return out
    lat = state["lat"]
    if case.get("job"):
        lat.init(*state["host"])
        lat.step(case["steps"])
        lbm.lbm_get_moments(lat.ctx, *[out[k] for k in FIELDS])
        return dict(out, totals=list(lat.totals()))
    lat.step(case["steps"])
    lbm.lbm_get_moments(lat.ctx, *[out[k] for k in FIELDS])
    return out


def work(case):
    """Bytes and operations of one pass: a step reads and writes every population and the phase-change
    history once, a read-out reads the populations and writes five fields."""
    n = sum(e[0] ** 3 for e in _instances(case)) if case["kind"] == "ensemble" else case["nx"] * case["ny"] * case["nz"]
    size = 4 if case.get("precision", "fp32") == "fp32" else 2
    pops = 19 + case.get("thermal_q", 7)
    step, read = 2 * pops * size + 8, pops * size + 20
    total = n * (case["steps"] * step + read)
    if case.get("job"):
        total += n * 20 + n * pops * size   # host fields in, first populations out
    return {"bytes": total, "flops": n * (case["steps"] * 650 + 150)}


# ----------------------------------------------------------------------------- the same in FP64
E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1)]
W19 = [1 / 3 if e == (0, 0, 0) else 1 / 18 if sum(map(abs, e)) == 1 else 1 / 36 for e in E]
WG = [0.0 if e == (0, 0, 0) else 1 / 6 if sum(map(abs, e)) == 1 else 1 / 12 for e in E]   # gradient weights
CS2 = 1.0 / 3.0


def _opp(a):
    return 0 if a == 0 else a + 1 if a % 2 else a - 1


def _moment_matrix():
    e = np.array(E, dtype=np.float64)
    x, y, z = e[:, 0], e[:, 1], e[:, 2]
    return np.stack([np.ones(19), x, y, z, x * x + y * y + z * z, 2 * x * x - y * y - z * z, y * y - z * z, x * y,
                     x * z, y * z, x * x * y, x * y * y, x * x * z, x * z * z, y * y * z, y * z * z, x * x * y * y,
                     x * x * z * z, y * y * z * z])


class _Exact:
    """One lattice in FP64: pull streaming, force, collisions and read-out with torch operations."""

    def __init__(self, case, rho, T, u):
        K = dict(KINDS["droplet" if case["kind"] == "ensemble" else case["kind"]])
        if case["kind"] == "ensemble":
            K.update(a=1 / 49, sigma=0.1175)
        self.K, self.dev = K, rho.device
        self.n = rho.shape[::-1]
        self.bc, self.Tc = K["bc"], _tc(K["a"])
        self.qt, self.divu_mode = case.get("thermal_q", 7), case.get("divu_mode", 0)
        self.wraps = [b in (PERIODIC, THERMAL) for b in self.bc]
        self.idx = {}
        for k in range(3):
            c = torch.arange(self.n[k], device=self.dev)
            for s in (-1, 1):
                q = c + s
                face = 2 * k + (s > 0)
                self.idx[k, s] = q % self.n[k] if self.wraps[face] else q.clamp(0, self.n[k] - 1)
        M = _moment_matrix()
        self.M = torch.tensor(M, device=self.dev)
        self.Mi = torch.tensor(np.linalg.inv(M), device=self.dev)
        d = 0.95
        self.csT2 = CS2 if self.qt == 19 else d / 3
        self.wg = W19 if self.qt == 19 else [1 - d] + [d / 6] * 6
        Tw = [t * self.Tc for t in K["Tw"]]
        x, y, _ = _grid(self.n[0], self.n[1], 1)
        self.Tw = [torch.full((self.n[1], self.n[0]), t, device=self.dev, dtype=torch.float64) for t in Tw]
        if "hot" in K:
            r2 = (x[0].double() - 0.5 * self.n[0]) ** 2 + (y[0].double() - 0.5 * self.n[1]) ** 2
            self.Tw[4] = self.Tw[4] + K["hot"] * self.Tc * torch.exp(-r2 / (2 * _hot_sigma(case) ** 2))
        if "wet" in K:
            h = _patch_half(case)
            inside = ((x[0] - 0.5 * self.n[0]).abs() < h) & ((y[0] - 0.5 * self.n[1]).abs() < h)
            p0, d0, p1, d1 = K["wet"]
            self.wphi = p0 + (p1 - p0) * inside.double()
            self.wdrho = d0 + (d1 - d0) * inside.double()
        rho, T = rho.double(), T.double()
        u = torch.zeros((3,) + rho.shape, device=self.dev, dtype=torch.float64) if u is None else u.double()
        self.f = self.transform(self.Mi, self.m_eq(rho, u))
        self.g = torch.stack([w * T for w in self.wg])
        self.mean, self.phis, self.fresh = float(rho.mean()), None, True

    def transform(self, A, v):
        return (A @ v.reshape(19, -1)).reshape(v.shape)

    def m_eq(self, r, u):
        x, y, z = u
        u2 = x * x + y * y + z * z
        phi = r * CS2 * CS2 * (1 - 1.5 * u2)
        return torch.stack([r, r * x, r * y, r * z, r + r * u2, r * (2 * x * x - y * y - z * z), r * (y * y - z * z),
                            r * x * y, r * x * z, r * y * z, r * y * (CS2 + x * x), r * x * (CS2 + y * y),
                            r * z * (CS2 + x * x), r * x * (CS2 + z * z), r * z * (CS2 + y * y),
                            r * y * (CS2 + z * z), phi + r * CS2 * (x * x + y * y), phi + r * CS2 * (x * x + z * z),
                            phi + r * CS2 * (y * y + z * z)])

    def shifted(self, A, s):
        """A at x + s, wrapped or clamped at the faces (the last three dimensions are z, y, x; or y, x)."""
        for k in range(3):
            if s[k]:
                A = A.index_select(A.dim() - 1 - k, self.idx[k, s[k]])
        return A

    def face(self, k, hi):
        return tuple([slice(None)] * (2 - k) + [-1 if hi else 0])

    def pulled(self):
        if self.fresh:
            return self.f, self.g
        f, g = torch.empty_like(self.f), torch.empty_like(self.g)
        for a, e in enumerate(E):
            f[a] = self.shifted(self.f[a], [-c for c in e])
            for k in range(3):
                if e[k] and self.bc[2 * k + (e[k] < 0)] == WALL:
                    at = self.face(k, e[k] < 0)
                    f[a][at] = self.f[_opp(a)][at]
        if self.K.get("thermal_off"):
            return f, self.g
        for a, e in enumerate(E[:self.qt]):
            g[a] = self.shifted(self.g[a], [-c for c in e])
            for k in range(3):
                face = 2 * k + (e[k] < 0)
                if e[k] and self.bc[face] != PERIODIC:
                    at = self.face(k, e[k] < 0)
                    Tw = self.Tw[face] if face == 4 else float(self.Tw[face][0, 0])
                    g[a][at] = -self.g[_opp(a)][at] + 2 * self.wg[a] * Tw
        return f, g

    def psi(self, rho, T):
        K = self.K
        kappa = 0.37464 + 1.54226 * ACENTRIC - 0.26992 * ACENTRIC ** 2
        theta = (1 + kappa * (1 - torch.sqrt(T / self.Tc))) ** 2
        br = B_EOS * rho
        p = rho * R_EOS * T / (1 - br) - K["a"] * theta * rho * rho / (1 + 2 * br - br * br)
        return torch.sqrt(2 * (rho * CS2 - p))

    def macroscopic(self):
        """Pulled populations, rho, T, psi, interaction force, grad rho, total force and u."""
        f, g = self.pulled()
        rho, T = f.sum(0), g.sum(0)
        psi = self.psi(rho, T)
        wall = None
        if "wet" in self.K:
            r0 = rho[0]
            near = sum(self.shifted(r0, s) for s in ((1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0)))
            ra = r0 / 3 + near / 6
            rw = torch.maximum(self.wphi * ra - self.wdrho, 0.1 * ra)
            wall = (self.psi(rw, self.Tw[4]), rw)
        Fm, grad = torch.zeros((3,) + rho.shape, device=self.dev, dtype=torch.float64), None
        grad = torch.zeros_like(Fm)
        for a in range(1, 19):
            e = E[a]
            qp, qr = self.shifted(psi, e), self.shifted(rho, e)
            if wall is not None and e[2] < 0:
                qp[0] = self.shifted(wall[0], (e[0], e[1], 0))
                qr[0] = self.shifted(wall[1], (e[0], e[1], 0))
            for k in range(3):
                if e[k]:
                    Fm[k] += WG[a] * e[k] * qp
                    grad[k] += WG[a] * e[k] * qr
        Fm *= psi
        F = Fm.clone()
        F[2] += (rho - (self.K.get("rho_buoy", 0.0) or self.mean)) * self.K.get("gz", 0.0)
        u = torch.stack([(sum(e[k] * f[a] for a, e in enumerate(E) if e[k]) + 0.5 * F[k]) / rho for k in range(3)])
        return f, g, rho, T, psi, Fm, grad, F, u

    def step(self):
        K = self.K
        f, g, rho, T, psi, Fm, grad, F, u = self.macroscopic()
        x, y, z = u
        Fx, Fy, Fz = F
        tau_e, sigma, cV = 1.25, K["sigma"], 5.0
        Fu = (F * u).sum(0)
        S4 = 2 * Fu + 6 * sigma * (Fm * Fm).sum(0) / (psi * psi * (tau_e - 0.5))
        S = torch.stack([torch.zeros_like(rho), Fx, Fy, Fz, S4, 2 * (2 * Fx * x - Fy * y - Fz * z),
                         2 * (Fy * y - Fz * z), Fx * y + Fy * x, Fx * z + Fz * x, Fy * z + Fz * y, CS2 * Fy, CS2 * Fx,
                         CS2 * Fz, CS2 * Fx, CS2 * Fz, CS2 * Fy, 2 * CS2 * (x * Fx + y * Fy),
                         2 * CS2 * (x * Fx + z * Fz), 2 * CS2 * (y * Fy + z * Fz)])
        m, me = self.transform(self.M, f), self.m_eq(rho, u)
        L = torch.tensor([1.0] * 4 + [1 / tau_e] + [1 / 0.8] * 5 + [1.0] * 9, device=self.dev, dtype=torch.float64)
        L = L[:, None, None, None]
        new_f = self.transform(self.Mi, m - L * (m - me) + (1 - 0.5 * L) * S)
        divu = (-(m[4] - me[4]) / tau_e + (1 - 0.5 / tau_e) * S4 - 2 * Fu) * 1.5 / rho
        if self.divu_mode:
            fd = sum(WG[a] * sum(e[k] * self.shifted(u[k], e) for k in range(3) if e[k]) for a, e in enumerate(E) if a)
            for k in range(3):
                for hi in (0, 1):
                    if not self.wraps[2 * k + hi]:
                        at = self.face(k, hi)
                        fd[at] = divu[at]
            divu = fd
        new_g = self.g
        if not K.get("thermal_off"):
            chi = K["chi"] / (rho * cV) if K.get("lambda_mode") else K.get("chi", 0.08) + 0 * rho
            vs = chi / self.csT2 + 0.5
            e = E[:self.qt]
            n = [sum(e[a][k] * g[a] for a in range(self.qt) if e[a][k]) for k in range(3)]
            gT = [-q / (vs * self.csT2) for q in n]
            phis = sum((chi * grad[k] / rho - u[k]) * gT[k] for k in range(3))
            phis = phis - T / (rho * cV) * (rho * R_EOS / (1 - B_EOS * rho)) * divu
            q = 1.5 * phis - 0.5 * (phis if self.phis is None else self.phis)
            self.phis = phis
            if self.qt == 19:
                new_g = torch.stack([g[a] - (g[a] - w * T) / vs + w * q for a, w in enumerate(self.wg)])
            else:   # MRT: first moments at 1 / vs, second moments at unit rates
                d = 0.95
                n1, n2, n3 = [v * (1 - 1 / vs) for v in n]
                n4 = d * T
                h = [T - n4, (n4 + 3 * n1) / 6, (n4 - 3 * n1) / 6, (n4 + 3 * n2) / 6, (n4 - 3 * n2) / 6,
                     (n4 + 3 * n3) / 6, (n4 - 3 * n3) / 6]
                new_g = torch.stack([h[a] + w * q for a, w in enumerate(self.wg)])
        self.mean = float(rho.mean())
        self.f, self.g, self.fresh = new_f, new_g, False

    def moments(self):
        _, _, rho, T, _, _, _, _, u = self.macroscopic()
        return dict(rho=rho, ux=u[0], uy=u[1], uz=u[2], T=T)


def exact(case, seed):
    if case["kind"] == "ensemble":
        if sum(e[0] ** 3 for e in _instances(case)) * case["steps"] > 4e8:
            return None
        parts = []
        for rho, T in _ensemble_fields(case, seed):
            s = _Exact(case, rho, T, None)
            for _ in range(case["steps"] + 1):   # prepare has taken one step
                s.step()
            parts.append(s.moments())
        return {k: torch.cat([p[k].ravel() for p in parts]) for k in FIELDS}
    s = _Exact(case, *_fields(case, seed))
    for _ in range(case["steps"]):
        s.step()
    out = s.moments()
    if case.get("precision", "fp32") != "fp32":
        # 16-bit storage: the rounding of the stored populations moves u by more than the flow's own
        # velocity in these runs, so only rho and T have a value to be held to
        out.update(ux=None, uy=None, uz=None)
    if case.get("job"):
        out["totals"] = [float(out["rho"].sum()), float(out["T"].sum()), s.mean]
    return out
