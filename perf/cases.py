"""Workloads of this package for performance measurements: inputs, one pass, its cost and its value.

Every case is work that a program using the package hands to its public entry points
(``sim.Simulation``, ``autograd.FdtdProbeLoss``, ``optimize.NormObjective``), at sizes of the
repository's experiments, tests and benchmark or between them:

  norm    one evaluation of the optimiser's objective (dispersion norm and its gradient)
  run     a field run: set the state, advance n steps (optionally with the rigid bunch, the
          absorbing layers and the field energy behind the bunch), read the state back
  waves   the dispersion measurement: one step, then the plane-wave amplitude, n times
  grad    loss and coefficient gradient of a probe-plane misfit through the autograd function
  batch   the same for a batch of independent 2D runs (checkpoints, recorded history, adjoint)
  pic     macro-particle cycles: a relativistic bunch, or an electron-ion plasma

``listed`` gives the named cases, ``draw`` one more from the same ranges, ``prepare`` what a
program holds before the call, ``run`` one pass, ``work`` the bytes and operations it cannot do
without, and ``exact`` its outputs in 64 bits, written with plain torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1710_06829_gb300 import _lib as L
from paper_1710_06829_gb300 import autograd as A
from paper_1710_06829_gb300 import optimize as O
from paper_1710_06829_gb300 import sim as S

DEV = "cuda"
DX = (1.0, 1.0, 1.0)
# coefficient sets as theta = (delta_x, delta_perp, beta_x, beta_perp): Yee, and the 3D lifts of
# Table 1's min.1, min.3 and Lehe schemes
SCHEMES = {"yee": (0.0, 0.0, 0.0, 0.0), "min1": (-0.125, -0.125, 0.110, 0.110),
           "min3": (-0.065, -0.065, -0.065, -0.065), "lehe": (-0.021, 0.0, 0.125, 0.0)}
TORCH = {"f32": torch.float32, "f64": torch.float64}
WEIGHTS = {"uniform": (L.FDTD_W_UNIFORM, 0.0), "cone": (L.FDTD_W_CONE_X, math.radians(30.0)),
           "gauss": (L.FDTD_W_GAUSS_Y, 0.1)}
SPONGE = 0.3      # strength of the absorbing layers
BUNCH = dict(q=1.0, v=0.999, sigma_par=4.0, sigma_perp=8.0)


# ---------------------------------------------------------------- cases

def _run(nx, ny, nz, dtype, scheme, steps, bunch=False, layer=0):
    return {"kind": "run", "nx": nx, "ny": ny, "nz": nz, "dtype": dtype, "scheme": scheme,
            "steps": steps, "bunch": bunch, "layer": layer}


def listed():
    return [
        # one objective evaluation of the 2D SLSQP searches (Table 1): the smallest call
        dict(name="norm2d_256", kind="norm", dims=2, nx=256, ny=256, nz=1, weight="uniform",
             scheme="min3"),
        # one objective evaluation of the 3D minimisation with the 30 degree cone weight
        dict(name="norm3d_256_cone", kind="norm", dims=3, nx=256, ny=256, nz=256, weight="cone",
             scheme="min3"),
        # the small 2D pulse run in 64 bits: a launch-bound time loop
        dict(name="te2d_128_f64", **_run(128, 128, 1, "f64", "min3", 200)),
        # a 2D run of ordinary, ragged size
        dict(name="te2d_1000x750_f32", **_run(1000, 750, 1, "f32", "min1", 100)),
        # the benchmark's 3D field run
        dict(name="vac3d_256_f32", **_run(256, 256, 256, "f32", "min3", 20)),
        # rigid bunch with absorbing layers in a radiation field, on a ragged grid (Cherenkov run)
        dict(name="bunch3d_300x250x225_f32", **_run(300, 250, 225, "f32", "min1", 50, True, 16)),
        # a 3D run in 64 bits
        dict(name="vac3d_192x128x96_f64", **_run(192, 128, 96, "f64", "min3", 20)),
        # phase-velocity measurement of a plane wave
        dict(name="waves3d_256_f32", kind="waves", nx=256, ny=256, nz=256, dtype="f32",
             scheme="min3", steps=20, mx=32, my=0, mz=0),
        # loss and gradient of the differentiable 3D run
        dict(name="grad3d_128_f32", kind="grad", nx=128, ny=128, nz=128, dtype="f32", steps=100,
             every=25),
        # loss and gradient of 32 independent 2D runs (propagation term of the optimiser)
        dict(name="grad2d_512x32_f32", kind="batch", nx=512, ny=512, batch=32, steps=64, every=32,
             scheme="min3"),
        # relativistic particle bunch with absorbing layers (Sec. 6) in a radiation field, the
        # largest grid
        dict(name="pic_bunch_512x256x256", kind="pic", plasma=False, nx=512, ny=256, nz=256,
             particles=1 << 22, layer=16, steps=16, scheme="min1", spread=0.0),
        # electron-ion plasma, two particles of each species in a cell, which have drifted about
        # a cell away from the cell order they were loaded in
        dict(name="pic_plasma_128", kind="pic", plasma=True, nx=128, ny=128, nz=128,
             particles=2, layer=0, steps=10, scheme="lehe", spread=1.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(rng, lo, hi, cells):
    """Three grid extents, log-uniform in [lo, hi], nx a multiple of 4, at most `cells` cells; half
    of them with x a multiple of 64 and y of 8 (a common choice), the others as they come."""
    while True:
        nx, ny, nz = (_log(rng, lo, hi) for _ in range(3))
        if rng.random() < 0.5:
            nx, ny = max(64, nx // 64 * 64), max(8, ny // 8 * 8)
        nx = max(4, nx // 4 * 4)
        if nx * ny * nz <= cells:
            return nx, ny, nz


def draw(rng):
    kind = rng.choice(["norm", "run2d", "run3d", "run3d", "waves", "grad", "batch", "bunch", "plasma"])
    scheme = rng.choice(["yee", "min1", "min3", "lehe"])
    if kind == "norm":
        weight = rng.choice(["uniform", "cone", "gauss"])
        if rng.random() < 0.5:
            return dict(kind="norm", dims=2, nx=_log(rng, 64, 1024), ny=_log(rng, 64, 1024), nz=1,
                        weight=weight, scheme=rng.choice(["yee", "min1", "min3"]))
        return dict(kind="norm", dims=3, nx=_log(rng, 24, 256), ny=_log(rng, 24, 256),
                    nz=_log(rng, 24, 256), weight=weight, scheme=scheme)
    if kind == "run2d":
        nx, ny, _ = _sizes(rng, 32, 2048, 1 << 30)
        return _run(nx, ny, 1, rng.choice(["f32", "f64"]), rng.choice(["yee", "min1", "min3"]),
                    _log(rng, 20, 200))
    if kind == "run3d":
        dtype = rng.choice(["f32", "f32", "f64"])
        nx, ny, nz = _sizes(rng, 32, 320, (1 << 24) if dtype == "f32" else (1 << 22))
        bunch = min(nx, ny, nz) >= 64 and rng.random() < 0.4
        layer = rng.choice([0, 8, 16]) if min(ny, nz) >= 48 else 0
        return _run(nx, ny, nz, dtype, scheme, _log(rng, 10, 50), bunch, layer)
    if kind == "waves":
        nx, ny, nz = _sizes(rng, 32, 256, 1 << 24)
        return dict(kind="waves", nx=nx, ny=ny, nz=nz, dtype=rng.choice(["f32", "f32", "f64"])
                    if nx * ny * nz <= 1 << 22 else "f32", scheme=scheme, steps=_log(rng, 5, 20),
                    mx=rng.randint(1, 16), my=rng.randint(0, 8), mz=rng.randint(0, 8))
    if kind == "grad":
        dtype = rng.choice(["f32", "f32", "f64"])
        nx, ny, nz = _sizes(rng, 32, 160, (1 << 21) if dtype == "f32" else (1 << 19))
        every = rng.choice([10, 25, 32])
        return dict(kind="grad", nx=nx, ny=ny, nz=nz, dtype=dtype, steps=_log(rng, 20, 100),
                    every=every)
    if kind == "batch":
        nx, ny, _ = _sizes(rng, 64, 512, 1 << 30)
        return dict(kind="batch", nx=nx, ny=ny, batch=_log(rng, 2, 32), steps=_log(rng, 16, 64),
                    every=rng.choice([16, 32]), scheme=rng.choice(["yee", "min1", "min3"]))
    if kind == "bunch":
        nx, ny, nz = _sizes(rng, 96, 512, 1 << 25)
        return dict(kind="pic", plasma=False, nx=nx, ny=ny, nz=nz, particles=_log(rng, 1 << 16, 1 << 22),
                    layer=rng.choice([0, 16]), steps=_log(rng, 4, 16), scheme=scheme, spread=0.0)
    nx, ny, nz = _sizes(rng, 32, 160, 1 << 21)
    return dict(kind="pic", plasma=True, nx=nx, ny=ny, nz=nz, particles=rng.randint(1, 4), layer=0,
                steps=_log(rng, 4, 10), scheme=scheme, spread=rng.choice([0.0, 1.0, 4.0]))


# ---------------------------------------------------------------- coefficients and inputs

def _theta(scheme):
    dx, dp, bx, bp = SCHEMES[scheme]
    beta = np.array([[0.0, bx, bx], [bx, 0.0, bp], [bx, bp, 0.0]])
    return beta, np.array([dx, dp, dp])


def _dims(case):
    return 2 if case["kind"] == "batch" or case.get("nz", 1) == 1 else 3


def _dt(beta, delta, dims):
    """0.95 of the CFL limit on a unit grid.  S is a quadratic in u_i in [0, 1] with non-negative
    u_i^2 coefficients (delta <= 0), so its maximum over the box is at a corner."""
    best = 0.0
    for m in range(1 << dims):
        u = [(m >> i) & 1 for i in range(dims)]
        s = sum(u) - sum(4.0 * delta[i] * u[i] for i in range(dims))
        s -= sum(4.0 * beta[i][j] * u[i] * u[j] for i in range(dims) for j in range(dims) if i != j)
        best = max(best, s)
    return 0.95 / math.sqrt(best)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _waves_field(shape, gen, dtype, axes):
    """A superposition of four plane waves of 8 to 64 cells plus noise of 1e-3: [nz, ny, nx]."""
    z, y, x = (torch.arange(n, device=DEV, dtype=torch.float64) for n in shape)
    out = 1e-3 * torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64)
    r = torch.rand((4, 5), generator=gen, device=DEV, dtype=torch.float64).cpu().numpy()
    for a in r:
        k = [2 * math.pi / (8.0 * 8.0 ** v) if ax < axes else 0.0 for ax, v in enumerate(a[:3])]
        ph = (k[0] * x)[None, None, :] + (k[1] * y)[None, :, None] + (k[2] * z)[:, None, None]
        out += (0.25 + 0.5 * a[3]) * torch.cos(ph + 2 * math.pi * a[4])
    return out.to(dtype)


def _fields(case, gen):
    """The six initial fields: TE (E_x, E_y, B_z) in 2D, all components in 3D; a plasma starts from
    zero, a bunch in a radiation field about as strong as its own."""
    if case.get("plasma"):
        return [None] * 6
    amp = 1e-3 if case.get("bunch") or case["kind"] == "pic" else 1.0
    dims = _dims(case)
    shape = (case.get("nz", case.get("batch", 1)), case["ny"], case["nx"])
    dt = TORCH[case.get("dtype", "f32")]
    want = (0, 1, 5) if dims == 2 else range(6)
    return [_waves_field(shape, gen, dt, dims).mul_(amp) if c in want else None for c in range(6)]


def _plane_wave(case, dtype, seed):
    """E_z = cos(k.r + phase) (staggered position of E_z), B = 0, seeded noise of 1e-3 on every E."""
    shape = (case["nz"], case["ny"], case["nx"])
    k = _kvec(case)
    z, y, x = (torch.arange(n, device=DEV, dtype=torch.float64) for n in shape)
    ph = (k[0] * x)[None, None, :] + (k[1] * y)[None, :, None] + (k[2] * (z + 0.5))[:, None, None]
    g = _gen(seed)
    p0 = float(torch.rand(1, generator=g, device=DEV, dtype=torch.float64)) * 2 * math.pi
    E = [1e-3 * torch.randn(shape, generator=g, device=DEV, dtype=torch.float64) for _ in range(3)]
    E[2] += torch.cos(ph + p0)
    return [e.to(dtype) for e in E] + [None] * 3


def _kvec(case):
    return [2 * math.pi * case["m" + a] / case["n" + a] for a in "xyz"]


def _particles(case, seed):
    """[(x, u, q, q/m)] of each species, float32 (3, n) arrays."""
    g = _gen(seed)
    n3 = (case["nx"], case["ny"], case["nz"])
    f64 = dict(device=DEV, dtype=torch.float64)
    box = torch.tensor(n3, **f64)[:, None]
    if not case["plasma"]:
        # gamma = 10 along +x, widths (4, 8, 8) cells, ordered by z cell, y cell, x
        n = case["particles"]
        c = torch.tensor([min(64.0, n3[0] / 4), n3[1] / 2, n3[2] / 2], **f64)[:, None]
        w = torch.tensor([4.0, 8.0, 8.0], **f64)[:, None]
        x = c + w * torch.randn((3, n), generator=g, **f64).clamp(-4.0, 4.0)
        x = x[:, torch.argsort(x[0])]
        x = x[:, torch.argsort(x[1].floor() + 4096.0 * x[2].floor(), stable=True)]
        u = torch.zeros((3, n), **f64)
        u[0] = math.sqrt(99.0)
        return [(x.float().contiguous(), u.float().contiguous(), -1.0 / n, -1.0)]
    ppc, out = case["particles"], []
    k, j, i = torch.meshgrid(*(torch.arange(n, **f64) for n in n3[::-1]), indexing="ij")
    cell = torch.stack([i.reshape(-1), j.reshape(-1), k.reshape(-1)]).repeat_interleave(ppc, dim=1)
    for q, qm, uth in ((-0.04 / ppc, -1.0, 0.1), (0.04 / ppc, 0.01, 0.01)):
        x = cell + torch.rand(cell.shape, generator=g, **f64)
        x = x + case["spread"] * torch.randn(cell.shape, generator=g, **f64)
        x = torch.remainder(x, box).float()
        x = torch.where(x >= box.float(), torch.zeros_like(x), x)
        u = uth * torch.randn(cell.shape, generator=g, **f64)
        out.append((x.contiguous(), u.float().contiguous(), q, qm))
    return out


def _norm_theta(case, seed):
    """The scheme's coefficients, moved by up to 1e-3 (a search's next point), and dt."""
    beta, delta = _theta(case["scheme"])
    r = np.random.default_rng(seed)
    for i in range(3):
        for j in range(i + 1, 3):
            beta[i, j] -= 1e-3 * r.uniform()
            beta[j, i] = beta[i, j]
    delta = delta - 1e-3 * r.uniform(size=3)
    d = case["dims"]
    b2, d2 = beta.copy(), delta.copy()
    b2[d:, :] = 0.0
    b2[:, d:] = 0.0
    d2[d:] = 0.0
    return b2, d2, _dt(b2, d2, d)


def _target(case, seed, nz):
    """Probe target [steps, nz, ny]: a smooth wave in time and along the plane."""
    g = _gen(seed + 7919)
    a = torch.rand(4, generator=g, device=DEV, dtype=torch.float64).cpu().numpy()
    s = torch.arange(1, case["steps"] + 1, device=DEV, dtype=torch.float64)[:, None, None]
    z = torch.arange(nz, device=DEV, dtype=torch.float64)[None, :, None]
    y = torch.arange(case["ny"], device=DEV, dtype=torch.float64)[None, None, :]
    t = torch.cos((0.1 + 0.1 * a[0]) * s + 0.05 * a[1] * y + 0.05 * a[2] * z + 6.0 * a[3])
    return t.to(TORCH[case.get("dtype", "f32")]).contiguous()


# ---------------------------------------------------------------- prepare and run

def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "norm":
        beta, delta, dt = _norm_theta(case, seed)
        w, p = WEIGHTS[case["weight"]]
        st["obj"] = O.NormObjective(list(DX), case["dims"], (case["nx"], case["ny"], case["nz"]), w, p)
        st["c"] = np.r_[beta.reshape(-1), delta, dt]
        return st
    dims = _dims(case)
    beta, delta = _theta("min3" if kind == "grad" else case["scheme"])
    dt = _dt(beta, delta, dims)
    if kind == "grad":
        shape = (case["nx"], case["ny"], case["nz"])
        st["theta"] = torch.tensor(SCHEMES["min3"], dtype=torch.float64)
        st["problem"] = A.ProbeLossProblem(
            shape, DX, dt, _fields(case, _gen(seed)), 2, (3 * case["nx"]) // 4,
            _target(case, seed, case["nz"]), case["steps"], case["every"], dims=dims,
            dtype=case["dtype"])
        return st
    nz = case["batch"] if kind == "batch" else case["nz"]
    layer = case.get("layer", 0)
    st["sim"] = S.Simulation((case["nx"], case["ny"], nz), DX, dt, beta, delta, dims=dims,
                             dtype=case.get("dtype", "f32"), absorb_cells=layer,
                             absorb_sigma=SPONGE if layer else 0.0, batched=kind == "batch")
    if kind == "run":
        st["fields"] = _fields(case, _gen(seed))
        st["bunch"] = S.Bunch(**_bunch(case, seed)) if case["bunch"] else None
    elif kind == "waves":
        st["fields"] = _plane_wave(case, TORCH[case["dtype"]], seed)
    elif kind == "batch":
        st["fields"] = _fields(case, _gen(seed))
        st["probe"] = S.Probe(1, (3 * case["nx"]) // 4, _target(case, seed, nz))
    else:
        st["fields"] = _fields(case, _gen(seed + 1))
        st["particles"] = _particles(case, seed)
    return st


def _bunch(case, seed):
    r = np.random.default_rng(seed).uniform(size=3)
    return dict(BUNCH, x0=case["nx"] / 4 + 4 * r[0], y0=case["ny"] / 2 + 4 * r[1],
                z0=case["nz"] / 2 + 4 * r[2])


def _window(case, x0, travel):
    """x-window of the field energy behind the bunch, and the margin to the layers."""
    return int(math.floor(x0 + travel - case["nx"] / 3)), case["nx"] // 4, case["layer"]


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "norm":
        value, grad = st["obj"](st["c"])
        return [value, grad]
    if kind == "grad":
        theta = st["theta"].clone().requires_grad_(True)
        beta, delta = A.tied_coefficients(theta)
        loss = A.FdtdProbeLoss.apply(beta, delta, st["problem"])
        loss.backward()
        return [loss.detach(), theta.grad]
    sm, n = st["sim"], case["steps"]
    if kind == "run":
        sm.set_state(st["fields"])
        sm.step(n, source=st["bunch"])
        out = []
        if st["bunch"] is not None:
            s = st["bunch"].s
            out.append(sm.energy(*_window(case, s.x0, s.v * sm.dt * n)))
        return out + sm.get_state()
    if kind == "waves":
        k = _kvec(case)
        amps = torch.empty((n + 1, 2), dtype=torch.float64, device=DEV)
        sm.set_state(st["fields"])
        for s in range(n + 1):
            sm.plane_wave(2, k, out=amps[s])
            if s < n:
                sm.step(1)
        return [amps] + sm.get_state()
    if kind == "batch":
        every = case["every"]
        segs = [min(every, n - s) for s in range(0, n, every)]
        loss = torch.zeros(1, dtype=torch.float64, device=DEV)
        grad = torch.zeros(12, dtype=torch.float64, device=DEV)
        sm.set_state(st["fields"])
        for slot, m in enumerate(segs):
            sm.checkpoint_save(slot)
            sm.step(m, probe=st["probe"], loss=loss)
        sm.set_adjoint(None)
        for slot in range(len(segs) - 1, -1, -1):
            sm.checkpoint_restore(slot)
            sm.step(segs[slot], record=True)
            sm.step_adjoint(segs[slot], grad, probe=st["probe"])
        return [loss, grad] + sm.get_adjoint()
    sm.set_state(st["fields"])
    sp = [S.Species(x.clone(), u.clone(), q, qm) for x, u, q, qm in st["particles"]]
    sm.pic_step(n, sp)
    out = sm.get_state()
    for s in sp:
        out += [s.x, s.u]
    return out


# ---------------------------------------------------------------- cost

def work(case):
    """Bytes: fields in and out once in every step (24 B and 24 B a cell in FP32), particles in and
    out once in every cycle, results once.  Operations: those of the update formulas."""
    kind = case["kind"]
    n3 = case["nx"] * case["ny"] * case.get("nz", case.get("batch", 1))
    if kind == "norm":
        return {"bytes": 8 * 3 * (case["nx"] + case["ny"] + case["nz"]) + 8 * 14, "flops": 60 * n3}
    e = 8 if case.get("dtype") == "f64" else 4
    steps = case["steps"]
    if kind == "run":
        return {"bytes": 12 * e * n3 * (steps + 1), "flops": 100 * n3 * steps}
    if kind == "waves":
        return {"bytes": n3 * e * (12 * (steps + 1) + (steps + 1)), "flops": n3 * (104 * steps + 4)}
    if kind in ("grad", "batch"):
        # forward, forward again with its E history, reverse (lambda in and out, E history in)
        return {"bytes": n3 * e * steps * (12 + 15 + 15), "flops": n3 * steps * (100 + 100 + 160)}
    p = case["particles"] * (2 * n3 if case["plasma"] else 1)
    return {"bytes": steps * (12 * e * n3 + 12 * e * p), "flops": steps * (100 * n3 + 400 * p)}


# ---------------------------------------------------------------- values in 64 bits

def _sh(F, axis, n):
    """F at +n cells along axis (0 = x, 1 = y, 2 = z), periodic."""
    return torch.roll(F, -n, 2 - axis)


class _Scheme:
    """The update equations in plain torch: extended D* in Faraday's law, Yee's D in Ampere's."""

    def __init__(self, beta, delta, dims):
        self.dims = dims
        self.d = [delta[a] if a < dims else 0.0 for a in range(3)]
        self.b = [[beta[a][c] if a != c and a < dims and c < dims else 0.0 for c in range(3)]
                  for a in range(3)]
        self.a = [1.0 - 2.0 * (self.b[i][0] + self.b[i][1] + self.b[i][2]) - 3.0 * self.d[i]
                  for i in range(3)]

    def dstar(self, a, F):
        if a >= self.dims:
            return torch.zeros_like(F)
        ax = _sh(F, a, 1) - F
        out = self.a[a] * ax + self.d[a] * (_sh(F, a, 2) - _sh(F, a, -1))
        for c in range(self.dims):
            if c != a:
                out = out + self.b[a][c] * (_sh(ax, c, 1) + _sh(ax, c, -1))
        return out

    def dback(self, a, F):
        return F - _sh(F, a, -1) if a < self.dims else torch.zeros_like(F)

    def faraday(self, E, B, dt):
        return [B[0] + dt * (self.dstar(2, E[1]) - self.dstar(1, E[2])),
                B[1] + dt * (self.dstar(0, E[2]) - self.dstar(2, E[0])),
                B[2] + dt * (self.dstar(1, E[0]) - self.dstar(0, E[1]))]

    def ampere(self, E, B, dt):
        return [E[0] + dt * (self.dback(1, B[2]) - self.dback(2, B[1])),
                E[1] + dt * (self.dback(2, B[0]) - self.dback(0, B[2])),
                E[2] + dt * (self.dback(0, B[1]) - self.dback(1, B[0]))]

    def step(self, E, B, dt):
        B = self.faraday(E, B, dt)
        return self.ampere(E, B, dt), B


def _state64(fields, shape):
    f = [torch.zeros(shape, dtype=torch.float64, device=DEV) if t is None else t.double() for t in fields]
    return f[:3], f[3:]


def _layer(n, width):
    f = torch.ones(n, dtype=torch.float64, device=DEV)
    for d in range(1, width + 1):
        f[width - d] = f[n - 1 - width + d] = 1.0 - SPONGE * (d / width) ** 3
    return f


def _sponge(case):
    w = case.get("layer", 0)
    if not w:
        return None
    return _layer(case["nz"], w)[:, None, None] * _layer(case["ny"], w)[None, :, None]


def _cdf_difference(a, b):
    """Phi(a) - Phi(b) of the standard normal distribution, without cancellation in the tails."""
    r = math.sqrt(0.5)
    s = torch.where(a + b > 0, -1.0, 1.0)
    lo, hi = torch.minimum(s * a, s * b), torch.maximum(s * a, s * b)
    return torch.sign(a - b) * 0.5 * (torch.special.erfc(-hi * r) - torch.special.erfc(-lo * r))


def _exact_run(case, seed):
    beta, delta = _theta(case["scheme"])
    dims = _dims(case)
    dt = _dt(beta, delta, dims)
    sch = _Scheme(beta, delta, dims)
    shape = (case["nz"], case["ny"], case["nx"])
    E, B = _state64(_fields(case, _gen(seed)), shape)
    sp = _sponge(case)
    prof = None
    if case["bunch"]:
        b = _bunch(case, seed)

        def cells(n, c):
            d = torch.arange(n, dtype=torch.float64, device=DEV) - c
            d = d - n * torch.floor(d / n + 0.5)
            return _cdf_difference((d + 0.5) / b["sigma_perp"], (d - 0.5) / b["sigma_perp"])
        prof = cells(case["nz"], b["z0"])[:, None, None] * cells(case["ny"], b["y0"])[None, :, None]
    for s in range(case["steps"]):
        E, B = E, sch.faraday(E, B, dt)
        if sp is not None:
            B = [t * sp for t in B]
        E = sch.ampere(E, B, dt)
        if prof is not None:
            nx, vdt = case["nx"], b["v"] * dt
            d = torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5 - (b["x0"] + vdt * s)
            d = d - nx * torch.floor(d / nx + 0.5)
            row = (b["q"] / dt) * _cdf_difference(d / b["sigma_par"], (d - vdt) / b["sigma_par"])
            E[0] = E[0] - dt * row[None, None, :] * prof
        if sp is not None:
            E = [t * sp for t in E]
    out = []
    if case["bunch"]:
        lo, length, m = _window(case, b["x0"], b["v"] * dt * case["steps"])
        i = torch.remainder(torch.arange(lo, lo + length, device=DEV), case["nx"])
        e = sum((t[m:case["nz"] - m, m:case["ny"] - m][:, :, i] ** 2).sum() for t in E + B)
        out.append((0.5 * e).reshape(1))
    return out + E + B


def _exact_waves(case, seed):
    beta, delta = _theta(case["scheme"])
    dt = _dt(beta, delta, 3)
    sch = _Scheme(beta, delta, 3)
    shape = (case["nz"], case["ny"], case["nx"])
    E, B = _state64(_plane_wave(case, TORCH[case["dtype"]], seed), shape)
    k = _kvec(case)
    z, y, x = (torch.arange(n, device=DEV, dtype=torch.float64) for n in shape)
    ph = (k[0] * x)[None, None, :] + (k[1] * y)[None, :, None] + (k[2] * (z + 0.5))[:, None, None]
    c, s = torch.cos(ph), -torch.sin(ph)
    amps = []
    for n in range(case["steps"] + 1):
        amps.append(torch.stack([(E[2] * c).sum(), (E[2] * s).sum()]))
        if n < case["steps"]:
            E, B = sch.step(E, B, dt)
    return [torch.stack(amps)] + E + B


def _exact_grad(case, seed):
    """Loss, coefficient gradients and (batch) the adjoint state: one step at a time, newest first,
    with torch's autograd through the step."""
    batch = case["kind"] == "batch"
    dims = _dims(case)
    beta0, delta0 = _theta("min3" if case["kind"] == "grad" else case["scheme"])
    dt = _dt(beta0, delta0, dims)
    nz = case["batch"] if batch else case["nz"]
    comp, xp = (1 if batch else 2), (3 * case["nx"]) // 4
    E, B = _state64(_fields(case, _gen(seed)), (nz, case["ny"], case["nx"]))
    tgt = _target(case, seed, nz).double()
    n, keep = case["steps"], max(1, int(math.sqrt(case["steps"])))
    sch = _Scheme(beta0.tolist(), delta0.tolist(), dims)
    saved, loss = {}, torch.zeros((), dtype=torch.float64, device=DEV)
    for s in range(n):
        if s % keep == 0:
            saved[s] = (E, B)
        E, B = sch.step(E, B, dt)
        loss = loss + ((E[comp][:, :, xp] - tgt[s]) ** 2).sum()
    bt = torch.tensor(beta0, device=DEV, requires_grad=True)
    dl = torch.tensor(delta0, device=DEV, requires_grad=True)
    gb, gd = torch.zeros_like(bt), torch.zeros_like(dl)
    lam = [torch.zeros_like(E[0]) for _ in range(6)]
    for s0 in sorted(saved, reverse=True):
        seg = [saved[s0]]
        for s in range(s0, min(s0 + keep, n)):
            seg.append(sch.step(*seg[-1], dt))
        for s in range(min(s0 + keep, n) - 1, s0 - 1, -1):
            after = seg[s - s0 + 1][0][comp][:, :, xp]
            lam[comp][:, :, xp] += 2.0 * (after - tgt[s])
            f = [t.detach().requires_grad_(True) for t in seg[s - s0][0] + seg[s - s0][1]]
            E1, B1 = _Scheme(bt, dl, dims).step(f[:3], f[3:], dt)
            g = torch.autograd.grad(E1 + B1, f + [bt, dl], lam, allow_unused=True)
            lam = [torch.zeros_like(v) if t is None else t.clone() for t, v in zip(g[:6], f)]
            gb, gd = gb + g[6], gd + g[7]
    if batch:
        return [loss.reshape(1), torch.cat([gb.reshape(-1), gd])] + lam
    gb, gd = gb.cpu(), gd.cpu()
    gt = torch.stack([gd[0], gd[1] + gd[2], gb[0, 1] + gb[1, 0] + gb[0, 2] + gb[2, 0], gb[1, 2] + gb[2, 1]])
    return [loss, gt]


def _nodes(g):
    """The two nodes around the grid coordinates g and their first-order weights."""
    f = torch.floor(g)
    return f.long(), (1.0 - (g - f), g - f)


def _gather(F, off, x, n3):
    ax = [_nodes(x[a] - off[a]) for a in range(3)]
    idx = [[torch.remainder(ax[a][0] + m, n3[a]) for m in range(2)] for a in range(3)]
    flat = F.reshape(-1)
    out = 0.0
    for a in range(2):
        for b in range(2):
            for c in range(2):
                at = (idx[2][c] * n3[1] + idx[1][b]) * n3[0] + idx[0][a]
                out = out + ax[0][1][a] * ax[1][1][b] * ax[2][1][c] * flat[at]
    return out


def _exact_pic(case, seed):
    beta, delta = _theta(case["scheme"])
    dt = _dt(beta, delta, 3)
    sch = _Scheme(beta, delta, 3)
    n3 = (case["nx"], case["ny"], case["nz"])
    sp = _sponge(case)
    E, B = _state64(_fields(case, _gen(seed + 1)), n3[::-1])
    species = [[x.double(), u.double(), q, qm] for x, u, q, qm in _particles(case, seed)]
    box = torch.tensor(n3, dtype=torch.float64, device=DEV)[:, None]
    offE = [(0.5, 0, 0), (0, 0.5, 0), (0, 0, 0.5)]
    offB = [(0, 0.5, 0.5), (0.5, 0, 0.5), (0.5, 0.5, 0)]
    for _ in range(case["steps"]):
        B1 = sch.faraday(E, B, dt)
        if sp is not None:
            B1 = [t * sp for t in B1]
        Bm = [0.5 * (p + q) for p, q in zip(B, B1)]
        J = [torch.zeros(n3[0] * n3[1] * n3[2], dtype=torch.float64, device=DEV) for _ in range(3)]
        for s in species:
            X, U = torch.empty_like(s[0]), torch.empty_like(s[1])
            for lo in range(0, s[0].shape[1], 1 << 20):
                x, u = s[0][:, lo:lo + (1 << 20)], s[1][:, lo:lo + (1 << 20)]
                h = 0.5 * s[3] * dt
                Ep = torch.stack([_gather(E[a], offE[a], x, n3) for a in range(3)])
                Bp = torch.stack([_gather(Bm[a], offB[a], x, n3) for a in range(3)])
                um = u + h * Ep
                t = h * Bp / torch.sqrt(1.0 + (um ** 2).sum(0))
                r = 2.0 * t / (1.0 + (t ** 2).sum(0))
                up = um + torch.linalg.cross(um, t, dim=0)
                u1 = um + torch.linalg.cross(up, r, dim=0) + h * Ep
                x1 = x + dt * u1 / torch.sqrt(1.0 + (u1 ** 2).sum(0))
                f = torch.floor(x)
                m = torch.arange(-1, 3, dtype=torch.float64, device=DEV)[:, None]
                S0 = [(1.0 - (x[a] - (f[a] + m)).abs()).clamp_min(0.0) for a in range(3)]
                D = [(1.0 - (x1[a] - (f[a] + m)).abs()).clamp_min(0.0) - S0[a] for a in range(3)]
                at = [torch.remainder(f[a].long() + m.long(), n3[a]) for a in range(3)]
                for a in range(3):
                    b, c = [(1, 2), (0, 2), (0, 1)][a]
                    run_ = torch.cumsum(D[a], 0)
                    for ib in range(4):
                        for ic in range(4):
                            w = (S0[b][ib] * S0[c][ic] + 0.5 * D[b][ib] * S0[c][ic]
                                 + 0.5 * S0[b][ib] * D[c][ic] + D[b][ib] * D[c][ic] / 3.0)
                            for ia in range(3):
                                k = [None] * 3
                                k[a], k[b], k[c] = at[a][ia], at[b][ib], at[c][ic]
                                v = -(s[2] / dt) * run_[ia] * w
                                J[a].index_add_(0, (k[2] * n3[1] + k[1]) * n3[0] + k[0], v)
                X[:, lo:lo + (1 << 20)] = torch.remainder(x1, box)
                U[:, lo:lo + (1 << 20)] = u1
            s[0], s[1] = X, U
        B = B1
        E = sch.ampere(E, B, dt)
        E = [e - dt * j.reshape(e.shape) for e, j in zip(E, J)]
        if sp is not None:
            E = [t * sp for t in E]
    out = E + B
    for s in species:
        out += [s[0], s[1]]
    return out


def _exact_norm(case, seed):
    """Norm and gradient by torch's autograd through the dispersion relation on the k-grid."""
    beta, delta, dt0 = _norm_theta(case, seed)
    d = case["dims"]
    N = [case["nx"], case["ny"], case["nz"]]
    bt = torch.tensor(beta, device=DEV, requires_grad=True)
    dl = torch.tensor(delta, device=DEV, requires_grad=True)
    dt = torch.tensor(dt0, dtype=torch.float64, device=DEV, requires_grad=True)
    k1 = [(torch.arange(N[a], dtype=torch.float64, device=DEV) + 0.5) * math.pi / N[a] for a in range(d)]
    pref = math.prod(math.pi / N[a] for a in range(d))
    total, grads = 0.0, [torch.zeros_like(bt), torch.zeros_like(dl), torch.zeros_like(dt)]
    for kz in (k1[2].split(32) if d == 3 else [None]):
        k = torch.meshgrid(*([k1[0], k1[1]] + ([kz] if d == 3 else [])), indexing="ij")
        s2 = [torch.sin(0.5 * t) ** 2 for t in k]
        c = [torch.cos(t) for t in k]
        alpha = [1.0 - 2.0 * bt[i].sum() + 2.0 * bt[i, i] - 3.0 * dl[i] for i in range(d)]
        S2 = 0.0
        for i in range(d):
            Ai = alpha[i] + dl[i] * (1.0 + 2.0 * c[i])
            for j in range(d):
                if j != i:
                    Ai = Ai + 2.0 * bt[i, j] * c[j]
            S2 = S2 + s2[i] * Ai
        kn = torch.sqrt(sum(t * t for t in k))
        w = 1.0
        if case["weight"] == "cone":
            w = (k[0] >= kn * math.cos(WEIGHTS["cone"][1])).double()
        elif case["weight"] == "gauss":
            w = torch.exp(-(k[1] / WEIGHTS["gauss"][1]) ** 2)
        f = pref * (w * ((2.0 / dt) * torch.asin(dt * torch.sqrt(S2)) - kn) ** 2).sum()
        g = torch.autograd.grad(f, [bt, dl, dt])
        total = total + float(f.detach())
        grads = [p + q for p, q in zip(grads, g)]
    gb = grads[0].cpu().numpy()
    gd = grads[1].cpu().numpy()
    for i in range(3):
        gb[i, i] = 0.0
        for j in range(3):
            if i >= d or j >= d:
                gb[i, j] = 0.0
        if i >= d:
            gd[i] = 0.0
    return [total, np.r_[gb.reshape(-1), gd, float(grads[2])]]


def exact(case, seed):
    return {"norm": _exact_norm, "run": _exact_run, "waves": _exact_waves, "grad": _exact_grad,
            "batch": _exact_grad, "pic": _exact_pic}[case["kind"]](case, seed)
