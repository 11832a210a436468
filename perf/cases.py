"""Performance cases: the calls that programs built on this library make, over the
range of grids, precisions, models and options they make them with.

Six kinds of call, each through the package's public entry points:

  step     a few time steps of one RK3 simulation, then its fields read back
  drop     the same for the two-phase (AB2, level set) simulation
  batch    a few steps of a batch of resident simulations, then every member's fields
  poisson  the fast Poisson solve alone
  rhs      the stress right-hand side alone
  monitor  the status, divergence residual and monitoring quantities of a state

``exact`` restates the method in 64-bit torch, apart from the library's code: the
same discretisation (staggered faces, WENO5, low-storage RK3, AB2, spectral
projection), written with whole-array shifts.
"""

import math

import numpy as np
import torch

from paper_1803_09563_gb300 import evp

TWO_PI = 2.0 * math.pi
STATE_FIELDS = [evp.EVP_U, evp.EVP_V, evp.EVP_W, evp.EVP_P] + [evp.EVP_BXX + c for c in range(6)]
DIAG = (True, False, False, True, False, True)


# ------------------------------------------------------------------------- cases
def _step(name, model, nx, ny, nz, walls, fp64, steps, dt, option="", re=100.0):
    return {"name": name, "kind": "step", "model": model, "nx": nx, "ny": ny, "nz": nz, "walls": walls, "fp64": fp64,
            "steps": steps, "dt": dt, "option": option, "re": re}


def listed():
    return [
        # a small box in double precision: validation runs and parameter scans, where launches count
        _step("box_32_fp64", "oldroyd_b", 32, 32, 32, False, True, 4, 1e-3, re=1.0),
        # an obstacle in a periodic box whose lengths are not powers of two, double precision
        _step("obstacle_72_fp64", "saramito", 72, 54, 48, False, True, 2, 4e-3, "obstacle"),
        # the elastoviscoplastic channel, the library's headline workload
        _step("channel_fp32", "saramito", 256, 128, 128, True, False, 2, 1e-2),
        # a channel of odd lengths with the implicit viscous option (small Reynolds numbers)
        _step("channel_implicit_fp32", "oldroyd_b", 96, 100, 72, True, False, 2, 2e-2, "implicit", re=20.0),
        # forced viscoelastic turbulence, the largest single simulation
        _step("turbulence_256_fp32", "fene_p", 256, 256, 256, False, False, 2, 1e-3, "abc", re=200.0),
        # a drop in an elastoviscoplastic fluid; ten steps hold one re-distancing
        {"name": "drop_fp32", "kind": "drop", "nx": 128, "ny": 256, "nz": 128, "fp64": False, "steps": 10, "dt": 1e-3},
        # the resident simulations of a server: several sizes advanced together
        {"name": "batch_mixed_fp32", "kind": "batch", "sizes": "32,32,32,48,48,48,64,64,64,96,96,128", "fp64": False,
         "steps": 2, "dt": 2e-3},
        # the Poisson solve: a channel, a box of odd lengths, and a small call where latency counts
        {"name": "poisson_channel_fp32", "kind": "poisson", "nx": 256, "ny": 128, "nz": 128, "walls": True, "fp64": False},
        {"name": "poisson_odd_fp32", "kind": "poisson", "nx": 144, "ny": 96, "nz": 108, "walls": False, "fp64": False},
        {"name": "poisson_small_fp64", "kind": "poisson", "nx": 24, "ny": 36, "nz": 48, "walls": False, "fp64": True},
        # the stress right-hand side for a caller's own time integrator, rows that are no multiple of 16 bytes
        {"name": "rhs_ragged_fp32", "kind": "rhs", "model": "saramito", "nx": 162, "ny": 75, "nz": 64, "walls": True,
         "fp64": False},
        # what a long run looks at between output intervals
        {"name": "monitor_fp32", "kind": "monitor", "model": "saramito", "nx": 256, "ny": 128, "nz": 128, "walls": True,
         "fp64": False},
    ]


_SMOOTH = sorted({2 ** a * 3 ** b for a in range(9) for b in range(5) if 16 <= 2 ** a * 3 ** b <= 256})


def _lengths(rng, cells, walls):
    """Grid lengths of at most ``cells`` cells in all, each between 16 and 256."""
    while True:
        nx = rng.choice([n for n in _SMOOTH if n % 2 == 0])
        ny = int(round(math.exp(rng.uniform(math.log(16), math.log(200))))) if walls else rng.choice(_SMOOTH)
        nz = rng.choice(_SMOOTH)
        if 8192 <= nx * ny * nz <= cells:
            return nx, ny, nz


def _time_step(nx, ny, nz, walls, option, re):
    """A time step that a run on this grid would take: a quarter of a cell per step at the
    largest velocities, within a quarter of the explicit viscous limit."""
    lx, ly, lz = _box(walls)
    hx, hy, hz = lx / nx, ly / ny, lz / nz
    dt = 0.25 * (min(hx / 1.5, hy / 0.5, hz / 0.5) if walls else min(hx, hy, hz))
    if option != "implicit":
        dt = min(dt, 0.25 * 2.5 * re / (4 * (hx ** -2 + hy ** -2 + hz ** -2)))
    return float("%.3g" % min(dt, 2e-2))


def _cells(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "drop", "batch", "poisson", "poisson", "rhs", "monitor"])
    if kind == "batch":
        sizes = ",".join(str(rng.choice([32, 48, 64, 96])) for _ in range(rng.randint(2, 10)))
        return {"kind": kind, "sizes": sizes, "fp64": False, "steps": 2, "dt": round(rng.uniform(1e-3, 3e-3), 5)}
    fp64 = rng.random() < 0.35
    walls = rng.random() < 0.5
    if kind == "drop":
        n = rng.choice([32, 48, 64, 96])
        m = rng.choice([n, 2 * n])
        return {"kind": kind, "nx": n, "ny": m, "nz": n, "fp64": fp64 and n <= 48, "steps": 10,
                "dt": round(rng.uniform(5e-4, 1e-3), 6)}
    if kind == "step":
        model = rng.choice(["oldroyd_b", "fene_p", "saramito"])
        nx, ny, nz = _lengths(rng, _cells(rng, 16384, 200e3 if fp64 else 6e6), walls)
        option = rng.choice(["", "", "", "obstacle", "implicit" if walls else "abc"])
        re = round(rng.uniform(20.0, 200.0), 1)
        case = _step("", model, nx, ny, nz, walls, fp64, 2, _time_step(nx, ny, nz, walls, option, re), option, re)
        return {k: v for k, v in case.items() if k != "name"}
    nx, ny, nz = _lengths(rng, _cells(rng, 16384, 300e3 if fp64 and kind != "poisson" else 6e6), walls)
    case = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "walls": walls, "fp64": fp64}
    if kind != "poisson":
        case["model"] = rng.choice(["oldroyd_b", "fene_p", "saramito"])
    return case


def work(case):
    """Bytes and operations of one pass.  An RK3 substep reads velocity (3), pressure
    (1) and B (6), and the histories (9) except in the first; it writes as many, the
    histories except in the last."""
    w = 8 if case["fp64"] else 4
    if case["kind"] == "batch":
        cells = sum(int(n) ** 3 for n in case["sizes"].split(","))
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    words, flops = {"step": (96, 5400), "batch": (96, 5400), "drop": (42, 2600), "poisson": (2, 75), "rhs": (15, 1250),
                    "monitor": (9, 60)}[case["kind"]]
    steps = case.get("steps", 1)
    return {"bytes": float(words) * w * cells * steps, "flops": float(flops) * cells * steps}


# ------------------------------------------------------------------------ inputs
class Geometry:
    def __init__(self, nx, ny, nz, walls, box):
        self.n = (nx, ny, nz)
        self.nx, self.ny, self.nz, self.walls = nx, ny, nz, bool(walls)
        self.lx, self.ly, self.lz = box
        self.dx, self.dy, self.dz = self.lx / nx, self.ly / ny, self.lz / nz
        self.shape = (nz, ny, nx)

    def grid(self):
        return evp.make_grid(self.nx, self.ny, self.nz, self.lx, self.ly, self.lz, self.walls)


def _noise(gen, geo, kmax, slope):
    """A smooth random field: white noise filtered to 1 <= |k| <= kmax with amplitude |k|^slope."""
    f = torch.fft.rfftn(torch.randn(geo.shape, generator=gen, device="cuda", dtype=torch.float64))
    k = [torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64) for n in (geo.nz, geo.ny)]
    kx = torch.arange(geo.nx // 2 + 1, device="cuda", dtype=torch.float64)
    mag = torch.sqrt(k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + kx[None, None, :] ** 2)
    amp = torch.where((mag >= 1) & (mag <= kmax), mag.clamp(min=1.0) ** slope, torch.zeros_like(mag))
    return torch.fft.irfftn(f * amp, s=geo.shape)


def _velocity(gen, geo, kmax, slope, size):
    """A discretely solenoidal velocity (curl of a random potential) of max-norm ``size``,
    on top of the laminar profile between walls."""
    ax, ay, az = (_noise(gen, geo, kmax, slope) for _ in range(3))
    if geo.walls:
        edge = (torch.arange(geo.ny, device="cuda", dtype=torch.float64) + 1) * (2.0 / geo.ny) - 1
        cell = edge - 1.0 / geo.ny
        env = ((1 - edge ** 2) ** 2)[None, :, None]
        ax, az, ay = ax * env, az * env, ay * ((1 - cell ** 2) ** 2)[None, :, None]

    def low(a, axis):
        return a - torch.roll(a, 1, dims=axis)
    u = low(az, 1) / geo.dy - low(ay, 0) / geo.dz
    v = low(ax, 0) / geo.dz - low(az, 2) / geo.dx
    w = low(ay, 2) / geo.dx - low(ax, 1) / geo.dy
    s = size / max(float(q.abs().max()) for q in (u, v, w))
    u, v, w = u * s, v * s, w * s
    if geo.walls:
        u = u + (1 - cell ** 2)[None, :, None]
    return u, v, w


def _conformation(gen, geo, scale, amp):
    """A smooth symmetric positive-definite B = scale (I + amp S)^2, max |S| = 1."""
    m = []
    for c in range(6):
        s = _noise(gen, geo, 3, -1.0)
        m.append(s * (amp / float(s.abs().max())) + (1.0 if DIAG[c] else 0.0))
    a, b, c, d, e, f = m
    return [scale * x for x in (a * a + b * b + c * c, a * b + b * d + c * e, a * c + b * e + c * f,
                                b * b + d * d + e * e, b * c + d * e + e * f, c * c + e * e + f * f)]


def _sphere(geo):
    """Signed distance to a sphere (centre and radius as the drop workload's) at cell centres."""
    r = [(torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h - 2.0
         for n, h in zip(geo.n, (geo.dx, geo.dy, geo.dz))]
    return torch.sqrt(r[0][None, None, :] ** 2 + r[1][None, :, None] ** 2 + r[2][:, None, None] ** 2) - 0.5


def _obstacle(geo):
    """Solid fractions of a smooth-edged sphere, at the u, v and w faces."""
    out = []
    for axis in range(3):
        d = [((torch.arange(n, device="cuda", dtype=torch.float64) + (1.0 if axis == q else 0.5)) / n - 0.5)
             for q, n in enumerate(geo.n)]
        r = torch.sqrt(d[0][None, None, :] ** 2 + d[1][None, :, None] ** 2 + d[2][:, None, None] ** 2)
        out.append(torch.clamp((0.22 - r) * geo.n[0] + 0.5, 0.0, 1.0))
    return out


def _box(walls):
    return (4.0 * math.pi, 2.0, TWO_PI) if walls else (TWO_PI, TWO_PI, TWO_PI)


def _physics(case):
    """Geometry, model and parameters (keywords of make_params) of a case."""
    kind = case["kind"]
    prec = evp.EVP_FP64 if case["fp64"] else evp.EVP_FP32
    if kind == "drop":
        geo = Geometry(case["nx"], case["ny"], case["nz"], False, (4.0, 4.0 * case["ny"] / case["nx"], 4.0))
        return geo, "saramito", dict(Re=10.0, Wi=1.0, beta=0.5, Bi=0.2, bi_def=1, mu_ratio=1.0, sigma=0.1, drho_g=1.0,
                                     reinit_every=10, reinit_iters=2, integrator=evp.EVP_AB2, precision=prec)
    walls = case.get("walls", False)
    geo = Geometry(case["nx"], case["ny"], case["nz"], walls, _box(walls))
    model = case.get("model", "oldroyd_b")
    re = case.get("re", 100.0)
    prm = dict(Re=re, Wi=1.0, beta=0.5, precision=prec)
    if model == "saramito":
        prm["Bi"] = 0.5
    if model == "fene_p":
        prm.update(L2=900.0, Wi=5.0, beta=0.9)
    if walls:
        prm["dpdx"] = 2.0 / re
    option = case.get("option", "")
    if option == "abc":
        prm.update(abc_amp=1.0, abc_k=2.0)
    if option == "obstacle":
        prm["penalization"] = 1
    if option == "implicit":
        prm["viscous_implicit"] = 1
    return geo, model, prm


def _fields(case, seed):
    """The initial fields of a simulation, in the case's precision: {field id: tensor}."""
    geo, model, prm = _physics(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dtype = torch.float64 if case["fp64"] else torch.float32
    out = {}
    if case["kind"] == "drop":
        vel = _velocity(gen, geo, 4, -2.0, 0.2)
        out[evp.EVP_PHI] = _sphere(geo)
        b = _conformation(gen, geo, 1.5, 0.4)
    else:
        fine = case.get("option", "") == "abc"
        vel = _velocity(gen, geo, 8, -2.5 if fine else -2.0, 1.0 if not geo.walls else 0.5)
        b = _conformation(gen, geo, 2.0, 0.5)
        if prm.get("penalization"):
            out.update(zip((evp.EVP_SOLID_X, evp.EVP_SOLID_Y, evp.EVP_SOLID_Z), _obstacle(geo)))
    p = _noise(gen, geo, 4, -1.0)
    out.update(zip(STATE_FIELDS, list(vel) + [p * (0.1 / float(p.abs().max()))] + b))
    return {f: a.to(dtype).contiguous() for f, a in out.items()}


def _simulation(case, seed):
    geo, model, prm = _physics(case)
    sim = evp.Simulation(geo.grid(), model, evp.make_params(**prm))
    fields = _fields(case, seed)
    evp.evp_set_fields(sim.handle, list(fields), list(fields.values()))
    return sim


def _members(case, seed):
    """The single-simulation cases of a batch's members, with their seeds."""
    models = ("saramito", "oldroyd_b", "saramito")
    return [({"kind": "step", "model": models[q % 3], "nx": int(n), "ny": int(n), "nz": int(n), "walls": False,
              "fp64": case["fp64"], "steps": case["steps"], "dt": case["dt"], "option": "", "re": 100.0}, seed * 64 + q)
            for q, n in enumerate(case["sizes"].split(","))]


def _rhs_field(case, seed):
    geo, _, _ = _physics(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    f = _noise(gen, geo, max(geo.n), -0.5)
    f = f - f.mean()
    return (f / f.std()).to(torch.float64 if case["fp64"] else torch.float32)


def prepare(case, seed):
    kind = case["kind"]
    dtype = torch.float64 if case["fp64"] else torch.float32
    if kind == "batch":
        batch = evp.Batch(evp.EVP_FP64 if case["fp64"] else evp.EVP_FP32)
        sims, outs = [], []
        for one, s in _members(case, seed):
            sim = _simulation(one, s)
            batch.admit(sim, one["dt"])
            sims.append(sim)
            outs.append(torch.empty((len(STATE_FIELDS),) + sim.shape, dtype=dtype, device="cuda"))
        return {"case": case, "batch": batch, "sims": sims, "outs": outs}
    if kind == "poisson":
        geo, model, prm = _physics(case)
        rhs = _rhs_field(case, seed)
        return {"case": case, "sim": evp.Simulation(geo.grid(), model, evp.make_params(**prm)), "rhs": rhs,
                "psi": torch.empty_like(rhs)}
    sim = _simulation(case, seed)
    if kind == "rhs":
        return {"case": case, "sim": sim, "rt": torch.empty((6,) + sim.shape, dtype=dtype, device="cuda")}
    if kind == "monitor":
        return {"case": case, "sim": sim}
    if kind == "step":
        evp.evp_set_graph(sim.handle, True)
    fields = STATE_FIELDS + ([evp.EVP_PHI] if kind == "drop" else [])
    return {"case": case, "sim": sim, "fields": fields,
            "outs": [torch.empty(sim.shape, dtype=dtype, device="cuda") for _ in fields]}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "poisson":
        evp.evp_poisson_solve(state["sim"].handle, state["rhs"], state["psi"])
        return [state["psi"]]
    if kind == "rhs":
        evp.evp_stress_rhs(state["sim"].handle, state["rt"])
        return [state["rt"][c] for c in range(6)]
    if kind == "monitor":
        code, bits, max_div = state["sim"].sync(raise_on_error=False)
        return {"code": code, "bits": bits, "residual": max_div} | state["sim"].diagnostics()
    if kind == "batch":
        for _ in range(case["steps"]):
            state["batch"].step()
        for sim, out in zip(state["sims"], state["outs"]):
            evp.evp_get_fields(sim.handle, STATE_FIELDS, list(out.unbind(0)))
        return state["outs"]
    for _ in range(case["steps"]):
        state["sim"].step(case["dt"])
    evp.evp_get_fields(state["sim"].handle, state["fields"], state["outs"])
    return state["outs"]


# ------------------------------------------------- the method in 64-bit torch
def _at(f, geo, kind, i=0, j=0, k=0):
    """f at index offset (i, j, k) from every cell; with walls ``kind`` gives the ghost
    rule in y: 'c' copies the nearest row, 'u' is odd about the wall, 'v' is zero outside."""
    if i:
        f = torch.roll(f, -i, dims=2)
    if k:
        f = torch.roll(f, -k, dims=0)
    if j and not geo.walls:
        return torch.roll(f, -j, dims=1)
    if j:
        n = geo.ny
        row = torch.arange(n, device=f.device) + j
        out = (row < 0) | (row >= n)
        src = row.clamp(0, n - 1)
        if kind == "u":
            src = torch.where(row < 0, -1 - row, torch.where(row >= n, 2 * n - 1 - row, row))
        sign = torch.ones(n, dtype=f.dtype, device=f.device)
        if kind != "c":
            sign[out] = -1.0 if kind == "u" else 0.0
        f = f[:, src, :] * sign[None, :, None]
    return f


def _weno(v1, v2, v3, v4, v5):
    q1 = v1 / 3 - 7 * v2 / 6 + 11 * v3 / 6
    q2 = -v2 / 6 + 5 * v3 / 6 + v4 / 3
    q3 = v3 / 3 + 5 * v4 / 6 - v5 / 6
    s1 = 13 / 12 * (v1 - 2 * v2 + v3) ** 2 + 0.25 * (v1 - 4 * v2 + 3 * v3) ** 2
    s2 = 13 / 12 * (v2 - 2 * v3 + v4) ** 2 + 0.25 * (v2 - v4) ** 2
    s3 = 13 / 12 * (v3 - 2 * v4 + v5) ** 2 + 0.25 * (3 * v3 - 4 * v4 + v5) ** 2
    a1, a2, a3 = 0.1 / (1e-6 + s1) ** 2, 0.6 / (1e-6 + s2) ** 2, 0.3 / (1e-6 + s3) ** 2
    return (a1 * q1 + a2 * q2 + a3 * q3) / (a1 + a2 + a3)


def _one_sided(f, geo, axis):
    """The left- and right-biased WENO5 derivatives along an axis."""
    h = (geo.dx, geo.dy, geo.dz)[axis]
    p = [_at(f, geo, "c", **{"ijk"[axis]: d}) for d in range(-3, 4)]
    d = [p[m + 1] - p[m] for m in range(6)]
    return _weno(*d[:5]) / h, _weno(*d[:0:-1]) / h


def _advect(f, geo, vel):
    """u . grad f, upwinded by the centre velocity."""
    out = torch.zeros_like(f)
    for axis in range(3):
        left, right = _one_sided(f, geo, axis)
        out += vel[axis] * torch.where(vel[axis] > 0, left, right)
    return out


def _centre_velocity(U, V, W, geo):
    return (0.5 * (U + _at(U, geo, "u", i=-1)), 0.5 * (V + _at(V, geo, "v", j=-1)), 0.5 * (W + _at(W, geo, "u", k=-1)))


def _component(a, b):
    return {(0, 0): 0, (0, 1): 1, (0, 2): 2, (1, 1): 3, (1, 2): 4, (2, 2): 5}[(min(a, b), max(a, b))]


class _Material:
    """The constants of a case (unit density)."""

    def __init__(self, model, prm):
        mu = 1.0 / prm["Re"]
        self.model, self.lam = model, prm["Wi"]
        self.mu_s, self.mu_p = prm["beta"] * mu, (1 - prm["beta"]) * mu
        self.tau_y = prm.get("Bi", 0.0) * (mu if prm.get("bi_def", 0) == 0 else 1.0)
        self.L2 = prm.get("L2", 0.0)

    def stress(self, B, mu_p=None):
        g = (self.mu_p if mu_p is None else mu_p) / self.lam
        F, a = (self.L2 / (self.L2 - B[0] - B[3] - B[5]), self.L2 / (self.L2 - 3)) if self.model == "fene_p" else (1.0, 1.0)
        return [g * (F * B[c] - (a if DIAG[c] else 0.0)) for c in range(6)]

    def magnitude(self, B, mu_p=None):
        g = (self.mu_p if mu_p is None else mu_p) / self.lam
        t = [g * (B[c] - (1.0 if DIAG[c] else 0.0)) for c in range(6)]
        m = (t[0] + t[3] + t[5]) / 3
        return torch.sqrt(0.5 * ((t[0] - m) ** 2 + (t[3] - m) ** 2 + (t[5] - m) ** 2) + t[1] ** 2 + t[2] ** 2 + t[4] ** 2)

    def closure(self, B, mu_p=None):
        if self.model == "fene_p":
            return self.L2 / (self.L2 - B[0] - B[3] - B[5]), self.L2 / (self.L2 - 3)
        if self.model == "saramito" and self.tau_y > 0:
            mag = self.magnitude(B, mu_p)
            F = torch.where(mag > 0, (1 - self.tau_y / torch.where(mag > 0, mag, torch.ones_like(mag))).clamp(min=0.0),
                            torch.zeros_like(mag))
            return F, F
        return 1.0, 1.0


def _stress_rhs(U, V, W, B, geo, mat, mu_p=None):
    vel = _centre_velocity(U, V, W, geo)
    kinds = ("u", "c", "u")
    h = (geo.dx, geo.dy, geo.dz)
    L = [[None] * 3 for _ in range(3)]
    for a, F in enumerate((U, V, W)):
        for b in range(3):
            s = "ijk"[b]
            if a == b:
                L[a][b] = (F - _at(F, geo, "v" if a == 1 else "u", **{s: -1})) / h[b]
            else:
                L[a][b] = (_at(vel[a], geo, kinds[a], **{s: 1}) - _at(vel[a], geo, kinds[a], **{s: -1})) / (2 * h[b])
    F, av = mat.closure(B, mu_p)
    out = []
    for c, (a, b) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))):
        rt = ((av if DIAG[c] else 0.0) - F * B[c]) / mat.lam - _advect(B[c], geo, vel)
        for q in range(3):
            rt = rt + L[a][q] * B[_component(q, b)] + B[_component(a, q)] * L[b][q]
        out.append(rt)
    return out


def _advection(U, V, W, geo):
    """div(uu) at the u, v and w faces."""
    vel = (U, V, W)
    kinds = ("u", "v", "u")
    h = (geo.dx, geo.dy, geo.dz)
    out = []
    for a in range(3):
        acc = 0.0
        for b in range(3):
            sa, sb = "ijk"[a], "ijk"[b]
            if a == b:
                hi = (0.5 * (vel[a] + _at(vel[a], geo, kinds[a], **{sa: 1}))) ** 2
                lo = (0.5 * (vel[a] + _at(vel[a], geo, kinds[a], **{sa: -1}))) ** 2
            else:
                hi = (0.5 * (vel[a] + _at(vel[a], geo, kinds[a], **{sb: 1}))
                      * 0.5 * (vel[b] + _at(vel[b], geo, kinds[b], **{sa: 1})))
                lo = (0.5 * (vel[a] + _at(vel[a], geo, kinds[a], **{sb: -1}))
                      * 0.5 * (_at(vel[b], geo, kinds[b], **{sb: -1}) + _at(vel[b], geo, kinds[b], **{sa: 1, sb: -1})))
            acc = acc + (hi - lo) / h[b]
        out.append(acc)
    return out


def _laplacian(f, geo, kind):
    h = (geo.dx, geo.dy, geo.dz)
    return sum((_at(f, geo, kind, **{s: 1}) - 2 * f + _at(f, geo, kind, **{s: -1})) / h[q] ** 2 for q, s in enumerate("ijk"))


def _edge(f, geo, a, b):
    """Mean over the four centres around the +1/2 edge of the axes a and b."""
    sa, sb = "ijk"[a], "ijk"[b]
    return 0.25 * (f + _at(f, geo, "c", **{sa: 1}) + _at(f, geo, "c", **{sb: 1}) + _at(f, geo, "c", **{sa: 1, sb: 1}))


def _edge_low(f, geo, a, b):
    """The same around the edge +1/2 in a and -1/2 in b."""
    sa, sb = "ijk"[a], "ijk"[b]
    return 0.25 * (f + _at(f, geo, "c", **{sa: 1}) + _at(f, geo, "c", **{sb: -1}) + _at(f, geo, "c", **{sa: 1, sb: -1}))


def _div_stress(t, geo):
    h = (geo.dx, geo.dy, geo.dz)
    out = []
    for a in range(3):
        acc = (_at(t[_component(a, a)], geo, "c", **{"ijk"[a]: 1}) - t[_component(a, a)]) / h[a]
        for b in range(3):
            if b != a:
                s = t[_component(a, b)]
                acc = acc + (_edge(s, geo, a, b) - _edge_low(s, geo, a, b)) / h[b]
        out.append(acc)
    return out


def _wall_operator(geo, kind):
    """Eigenvalues and vectors of the wall-normal second difference (negated)."""
    n = geo.ny
    A = 2 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1)
    if kind == "c":
        A[0, 0] = A[-1, -1] = 1.0
    elif kind == "u":
        A[0, 0] = A[-1, -1] = 3.0
    else:   # the last stored face is the wall
        A = A[:-1, :-1]
    lam, Q = np.linalg.eigh(A / geo.dy ** 2)
    return torch.from_numpy(lam).cuda(), torch.from_numpy(np.ascontiguousarray(Q)).cuda()


def _solve(r, geo, kind="c", c=None):
    """psi of lap psi = r, or (with c) x of x - c lap x = r, for fields with ghost rule ``kind``."""
    def lam(n, h, count=None):
        m = torch.arange(n if count is None else count, device="cuda", dtype=torch.float64)
        return (2 - 2 * torch.cos(TWO_PI * m / n)) / h ** 2
    lx, lz = lam(geo.nx, geo.dx, geo.nx // 2 + 1), lam(geo.nz, geo.dz)
    if not geo.walls:
        f = torch.fft.rfftn(r)
        s = lx[None, None, :] + lam(geo.ny, geo.dy)[None, :, None] + lz[:, None, None]
        if c is not None:
            return torch.fft.irfftn(f / (1 + c * s), s=geo.shape)
        s[0, 0, 0] = 1.0
        f = -f / s
        f[0, 0, 0] = 0.0
        return torch.fft.irfftn(f, s=geo.shape)
    ly, Q = _wall_operator(geo, kind)
    f = torch.fft.rfftn(r, dim=(0, 2))
    if kind == "v":
        f = f[:, :-1, :]
    if c is None:   # the first row of the mean mode is replaced by psi = 0
        f[0, 0, 0] = -f[0, 1:, 0].sum()

    def modes(M, x):
        return torch.complex(torch.matmul(M, x.real.contiguous()), torch.matmul(M, x.imag.contiguous()))
    f = modes(Q.T.contiguous(), f)
    s = lx[None, None, :] + ly[None, :, None] + lz[:, None, None]
    if c is not None:
        f = modes(Q, f / (1 + c * s))
        if kind == "v":
            f = torch.cat([f, torch.zeros_like(f[:, :1, :])], 1)
        return torch.fft.irfftn(f, s=(geo.nz, geo.nx), dim=(0, 2))
    s[0, 0, 0] = 1.0
    f = -f / s
    f[0, 0, 0] = 0.0
    f = modes(Q, f)
    f[0, :, 0] -= f[0, 0, 0].clone()
    return torch.fft.irfftn(f, s=(geo.nz, geo.nx), dim=(0, 2))


def _divergence(U, V, W, geo):
    return ((U - _at(U, geo, "u", i=-1)) / geo.dx + (V - _at(V, geo, "v", j=-1)) / geo.dy
            + (W - _at(W, geo, "u", k=-1)) / geo.dz)


def _gradient(p, geo):
    return [(_at(p, geo, "c", **{s: 1}) - p) / h for s, h in zip("ijk", (geo.dx, geo.dy, geo.dz))]


def _no_wall_flux(V, geo):
    if geo.walls:
        V = V.clone()
        V[:, -1, :] = 0.0
    return V


def _exact_steps(case, fields):
    """``steps`` RK3 steps from the given fields."""
    geo, model, prm = _physics(case)
    mat = _Material(model, prm)
    U, V, W, p, *B = [fields[f].double() for f in STATE_FIELDS]
    V = _no_wall_flux(V, geo)
    solid = [fields[f].double() for f in (evp.EVP_SOLID_X, evp.EVP_SOLID_Y, evp.EVP_SOLID_Z)] if prm.get("penalization") else None
    force = [prm.get("dpdx", 0.0), 0.0, 0.0]
    if prm.get("abc_amp"):
        a, k = prm["abc_amp"], prm["abc_k"]
        x, y, z = ((torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h * k
                   for n, h in zip(geo.n, (geo.dx, geo.dy, geo.dz)))
        x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
        force = [force[0] + a * (torch.sin(z) + torch.cos(y)), a * (torch.sin(x) + torch.cos(z)),
                 a * (torch.sin(y) + torch.cos(x))]
    kinds = ("u", "v", "u")
    implicit = bool(prm.get("viscous_implicit"))
    dt = case["dt"]
    for _ in range(case["steps"]):
        rt_old = n_old = None
        for al, ze, xi in ((4 / 15, 8 / 15, 0.0), (1 / 15, 5 / 12, -17 / 60), (1 / 6, 3 / 4, -5 / 12)):
            rt = _stress_rhs(U, V, W, B, geo, mat)
            Bn = [B[c] + dt * (ze * rt[c] + (xi * rt_old[c] if xi else 0.0)) for c in range(6)]
            t = [x + y for x, y in zip(mat.stress(Bn), mat.stress(B))]
            adv, dtau, gp = _advection(U, V, W, geo), _div_stress(t, geo), _gradient(p, geo)
            lap = [_laplacian(f, geo, q) for f, q in zip((U, V, W), kinds)]
            N = [-adv[q] + (0.0 if implicit else mat.mu_s * lap[q]) + force[q] for q in range(3)]
            star = []
            for q, f in enumerate((U, V, W)):
                inc = ze * N[q] + (xi * n_old[q] if xi else 0.0) - 2 * al * gp[q] + al * dtau[q]
                if implicit:
                    inc = inc + al * mat.mu_s * lap[q]
                s = f + dt * inc
                if solid:
                    s = s * (1 - solid[q])
                star.append(s)
            star[1] = _no_wall_flux(star[1], geo)
            if implicit:
                star = [_solve(s, geo, q, al * dt * mat.mu_s) for s, q in zip(star, kinds)]
            psi = _solve(_divergence(*star, geo) / (2 * al * dt), geo)
            g = _gradient(psi, geo)
            U, V, W = (s - 2 * al * dt * x for s, x in zip(star, g))
            V = _no_wall_flux(V, geo)
            p = p + psi
            B, rt_old, n_old = Bn, rt, N
    return [U, V, W, p] + B


def _exact_drop(case, fields):
    """``steps`` two-phase AB2 steps (periodic box, Boussinesq drop) from the given fields."""
    geo, model, prm = _physics(case)
    mat = _Material(model, prm)
    U, V, W, p, *B = [fields[f].double() for f in STATE_FIELDS]
    phi = fields[evp.EVP_PHI].double()
    dt, dx, eps = case["dt"], geo.dx, 1.5 * geo.dx

    def tvd(f, rhs, h):
        a = f + h * rhs(f)
        b = 0.75 * f + 0.25 * (a + h * rhs(a))
        return f / 3 + 2 / 3 * (b + h * rhs(b))

    def central(f, s, h):
        return (_at(f, geo, "c", **{s: 1}) - _at(f, geo, "c", **{s: -1})) / (2 * h)
    h3 = (geo.dx, geo.dy, geo.dz)
    rt_old = n_old = None
    for step in range(case["steps"]):
        vel = _centre_velocity(U, V, W, geo)
        phi = tvd(phi, lambda f: -_advect(f, geo, vel), dt)
        if (step + 1) % prm["reinit_every"] == 0:
            sign = phi / torch.sqrt(phi ** 2 + dx ** 2)

            def distance(f):
                acc = torch.zeros_like(f)
                for axis in range(3):
                    left, right = _one_sided(f, geo, axis)
                    pos = torch.maximum(left.clamp(min=0) ** 2, right.clamp(max=0) ** 2)
                    neg = torch.maximum(left.clamp(max=0) ** 2, right.clamp(min=0) ** 2)
                    acc += torch.where(sign > 0, pos, neg)
                return -sign * (torch.sqrt(acc) - 1)
            for _ in range(prm["reinit_iters"]):
                phi = tvd(phi, distance, 0.5 * dx)
        H = torch.where(phi < -eps, torch.zeros_like(phi),
                        torch.where(phi > eps, torch.ones_like(phi),
                                    0.5 * (1 + phi / eps + torch.sin(math.pi * phi / eps) / math.pi)))
        g = [central(phi, s, h) for s, h in zip("ijk", h3)]
        mag = torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2).clamp(min=1e-12)
        n = [x / mag for x in g]
        kappa = -sum(central(x, s, h) for x, s, h in zip(n, "ijk", h3))
        delta = torch.where(phi.abs() > eps, torch.zeros_like(phi), 0.5 / eps * (1 + torch.cos(math.pi * phi / eps)))
        f = [prm["sigma"] * kappa * delta * x for x in n]
        f[1] = f[1] + ((1 - H) - (1 - H).mean()) * prm["drho_g"]
        mu_p = mat.mu_p * H
        mu = mat.mu_s * H + prm["mu_ratio"] / prm["Re"] * (1 - H)
        w1, w0 = (1.0, 0.0) if step == 0 else (1.5, -0.5)
        rt = _stress_rhs(U, V, W, B, geo, mat, mu_p)
        t = mat.stress(B, mu_p)
        # the viscous stress 2 mu D: normal parts at centres, shear parts at edges
        F = (U, V, W)
        visc = []
        for a in range(3):
            s = "ijk"[a]
            normal = 2 * mu * (F[a] - _at(F[a], geo, "u", **{s: -1})) / h3[a]
            acc = (_at(normal, geo, "c", **{s: 1}) - normal) / h3[a]
            for b in range(3):
                if b != a:
                    sb = "ijk"[b]
                    shear = _edge(mu, geo, a, b) * ((_at(F[a], geo, "u", **{sb: 1}) - F[a]) / h3[b]
                                                    + (_at(F[b], geo, "u", **{s: 1}) - F[b]) / h3[a])
                    acc = acc + (shear - _at(shear, geo, "c", **{sb: -1})) / h3[b]
            visc.append(acc)
        adv, dtau = _advection(U, V, W, geo), _div_stress(t, geo)
        N = [-adv[q] + visc[q] + dtau[q] + 0.5 * (f[q] + _at(f[q], geo, "c", **{"ijk"[q]: 1})) for q in range(3)]
        star = [F[q] + dt * (w1 * N[q] + (w0 * n_old[q] if w0 else 0.0)) for q in range(3)]
        B = [B[c] + dt * (w1 * rt[c] + (w0 * rt_old[c] if w0 else 0.0)) for c in range(6)]
        p = _solve(_divergence(*star, geo) / dt, geo)
        U, V, W = (s - dt * x for s, x in zip(star, _gradient(p, geo)))
        rt_old, n_old = rt, N
    return [U, V, W, p] + B + [phi]


def exact(case, seed):
    kind = case["kind"]
    geo, model, prm = _physics(case) if kind != "batch" else (None, None, None)
    if kind == "batch":
        return [torch.stack(_exact_steps(one, _fields(one, s))) for one, s in _members(case, seed)]
    if kind == "poisson":
        return [_solve(_rhs_field(case, seed).double(), geo)]
    fields = _fields(case, seed)
    if kind == "step":
        return _exact_steps(case, fields)
    if kind == "drop":
        return _exact_drop(case, fields)
    U, V, W, _, *B = [fields[f].double() for f in STATE_FIELDS]
    V = _no_wall_flux(V, geo)
    mat = _Material(model, prm)
    if kind == "rhs":
        return _stress_rhs(U, V, W, B, geo, mat)
    div = float(_divergence(U, V, W, geo).abs().max())
    det = (B[0] * (B[3] * B[5] - B[4] ** 2) - B[1] * (B[1] * B[5] - B[4] * B[2]) + B[2] * (B[1] * B[4] - B[3] * B[2]))
    tr = float((B[0] + B[3] + B[5]).max())
    cells = int((mat.magnitude(B) > mat.tau_y).sum()) if model == "saramito" else U.numel()
    if case["fp64"]:
        div = None   # the residual of a solenoidal field in double precision is its rounding
    return {"code": None, "bits": None, "residual": div,
            "kinetic_energy": float(0.5 * geo.dx * geo.dy * geo.dz * (U ** 2 + V ** 2 + W ** 2).sum()), "max_div": div,
            "min_det_B": float(det.min()), "max_tr_B": tr, "max_tr_B_over_L2": tr / mat.L2 if model == "fene_p" else 0.0,
            "yielded_fraction": cells / U.numel(), "nonfinite_cells": 0, "yielded_cells": cells}
