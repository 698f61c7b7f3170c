"""The work a user of the library has it do, as cases to time and compare.

Every case goes through the public entry points: the ``Simulation`` binding
and the C-ABI of include/picsar.h (with device buffers where a GPU program
would read results on the device).  The grids, plasmas and physics are those
of the repository's workloads (the monopole plasmas, the monopole rotator with
surface injection, the uneven ensemble), on sizes from a few thousand cells to
four million and from some ten thousand particles to a quarter of a billion.

Results of the FP32 path are handed on in FP32, the precision that path holds
and computes its particles in; results of the FP64 path in FP64.  FP64
particles are returned too (that path keeps them in load and injection order).

``exact`` restates the method in plain torch FP64 operations.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

from paper_1407_1810_gb300 import picsar as P

DEV = "cuda"

# ---- the families of workloads ----------------------------------------------
# a pair plasma around a vacuum monopole on a log-r, linear-theta grid
MONOPOLE = dict(r_min=1.0, r_max=100.0, r_map="log", th_map="linear", courant=0.5, n_filt=0, absorb_cells=32,
                absorb_profile="linear", vacuum="monopole", omega=0.0, t_spin=0.0, inject=0, inject_pairs=2,
                f_inj=0.0, inject_smooth=0, pusher="vay", T=0.3, wc_dt=0.5, wp_dt=0.05, sort_interval=20)
# the rotating monopole with surface injection, three filter passes and a
# quadratic lossy layer on a log-r, equal-area grid
ROTATOR = dict(r_min=1.0, r_max=40.0, r_map="log", th_map="equal_area", courant=0.5, n_filt=3, absorb_cells=32,
               absorb_profile="quadratic", vacuum="monopole_rotator", omega=0.2, t_spin=0.5 * 2 * math.pi / 0.2,
               inject=1, inject_pairs=2, f_inj=0.5, inject_smooth=0, pusher="vay", T=0.1, wc_dt=4.0, wp_dt=0.05,
               sort_interval=20)
# an aligned dipole rotator with the paper's variable-count injection, one
# smoothing and one filter pass, Boris pusher, linear theta: the FP32 path's
# general form (no compile-time specialisation)
DIPOLE = dict(ROTATOR, th_map="linear", n_filt=1, absorb_cells=16, absorb_profile="linear", vacuum="dipole_rotator",
              inject=2, inject_pairs=4, inject_smooth=1, pusher="boris", wc_dt=1.0)
FAMILY = {"monopole": MONOPOLE, "rotator": ROTATOR, "dipole": DIPOLE}


def listed():
    return [
        # the smallest calls: a study on a coarse grid with injection, FP64 and
        # FP32, where launches and latency count (the test suite's rotator sizes)
        dict(name="rotator-64-fp64", do="steps", family="rotator", precision="fp64", nr=64, nth=64, pairs=12, steps=20,
             r_max=10.0, absorb_cells=8),
        dict(name="rotator-72x56-fp32", do="steps", family="rotator", precision="fp32", nr=72, nth=56, pairs=12,
             steps=20, r_max=10.0, absorb_cells=8),
        # the general kernel: dipole rotator, Boris, variable-count injection
        dict(name="dipole-192x160-fp32", do="steps", family="dipole", precision="fp32", nr=192, nth=160, pairs=10,
             steps=20),
        # an ordinary plain FP64 run on an odd-sized grid
        dict(name="monopole-200x163-fp64", do="steps", family="monopole", precision="fp64", nr=200, nth=163, pairs=12,
             steps=20),
        # an ordinary FP32 run: few tiles, two million particles
        dict(name="monopole-250x231-fp32", do="steps", family="monopole", precision="fp32", nr=250, nth=231, pairs=18,
             steps=20),
        # the FP64 rotator workload: 512 x 512, 2e7 particles, injection
        dict(name="rotator-512-fp64", do="steps", family="rotator", precision="fp64", nr=512, nth=512, pairs=38,
             steps=5),
        # the large run's plasma on 1024 x 1024: 6.3e7 particles, one sort cycle
        dict(name="monopole-1024-fp32", do="steps", family="monopole", precision="fp32", nr=1024, nth=1024, pairs=30,
             steps=20),
        # the FP32 rotator workload: 1024 x 1024, 1e8 particles
        dict(name="rotator-1024-fp32", do="steps", family="rotator", precision="fp32", nr=1024, nth=1024, pairs=48,
             steps=20),
        # the largest: 2048 x 2048, 2.5e8 particles
        dict(name="monopole-2048-fp32", do="steps", family="monopole", precision="fp32", nr=2048, nth=2048, pairs=30,
             steps=5),
        # the 64 uneven monopole plasmas advanced together
        dict(name="ensemble-64", do="ensemble", members=64, n_lo=1e4, n_hi=2e6, steps=40),
        # a whole run as a script makes it: grid, load from pinned host
        # arrays, one sort cycle, fields
        dict(name="whole-run-448x416-fp32", do="whole", family="monopole", precision="fp32", nr=448, nth=416, pairs=20,
             steps=20),
        # the diagnostics of a running simulation: energies and Gauss law,
        # filtered charge density, luminosity profile
        dict(name="diagnostics-1024-fp32", do="diagnose", family="rotator", precision="fp32", nr=1024, nth=1024,
             pairs=24, steps=2),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    do = rng.choice(["steps"] * 8 + ["ensemble", "whole", "diagnose"])
    if do == "ensemble":
        return dict(do=do, members=rng.randint(5, 64), n_lo=1e4, n_hi=_log(rng, 1e5, 2e6), steps=40)
    kind = rng.choice(["rotator", "monopole"]) if do != "steps" else rng.choice(
        ["rotator", "monopole", "rotator", "monopole", "dipole"])
    prec = rng.choice(["fp32", "fp32", "fp64"]) if do == "steps" else "fp32"
    if prec == "fp64" and kind == "dipole":
        kind = "rotator"
    # grids from a few thousand cells up to the family's largest, any aspect
    # ratio up to two, odd sizes among them
    side = {"rotator": (48, 640), "monopole": (200, 768), "dipole": (96, 512)}[kind]
    n = _log(rng, *side)
    a = rng.uniform(0.7, 1.4)
    nr, nth = max(40, int(n * a)), max(40, int(n / a))
    pairs = rng.randint(4, 40)
    c = dict(do=do, family=kind, precision=prec, nr=nr, nth=nth, pairs=pairs, steps=20)
    if do == "diagnose":
        c["steps"] = 2
    elif prec == "fp64" and nr * nth * pairs * 2 > 4e6:
        c["steps"] = 5
    if kind == "rotator" and n < 150:
        c.update(r_max=10.0, absorb_cells=8)
    return c


# ---- set-up -------------------------------------------------------------------
def _config(case):
    f = dict(FAMILY[case["family"]])
    f.update({k: v for k, v in case.items() if k not in ("name", "do", "family")})
    return f


def _fr(f, x):
    if f["r_map"] == "log":
        return f["r_min"] * np.exp(x * (math.log(f["r_max"] / f["r_min"]) / f["nr"]))
    return f["r_min"] + x * ((f["r_max"] - f["r_min"]) / f["nr"])


def _fth(f, x):
    x = np.clip(x, 0.0, f["nth"])
    return np.arccos(1.0 - 2.0 * x / f["nth"]) if f["th_map"] == "equal_area" else math.pi * x / f["nth"]


def _physics(f):
    """Time step at the Courant number, field strength and macro-charge from
    the cyclotron and plasma frequencies at the star's equator."""
    r = _fr(f, np.arange(f["nr"] + 1.0))
    th = _fth(f, np.arange(f["nth"] + 1.0))
    dt = f["courant"] * float(min(np.diff(r).min(), (r[:-1] * np.diff(th).min()).min()))
    j = f["nth"] // 2
    vol = 2 * math.pi / 3 * (r[1] ** 3 - r[0] ** 3) * (math.cos(th[j - 1]) - math.cos(th[j]))
    qw = (f["wp_dt"] / dt) ** 2 * vol / (2 * max(f["pairs"], 1))
    if f["precision"] == "fp32":
        qw = float(np.float32(qw))
    # variable-count injection: about three pairs per cell from the vacuum surface charge
    b0 = f["wc_dt"] / dt
    dA = 2 * math.pi * f["r_min"] ** 2 * (math.cos(th[j - 1]) - math.cos(th[j]))
    inject_q = f["f_inj"] * b0 * f["omega"] * f["r_min"] * dA / 3.0 if f["inject"] == 2 else 0.0
    return dt, b0, qw, float(np.float32(inject_q))


def _capacity(f, n):
    """Particle slots: the plasma, and on a small grid the thousands of steps of
    injection that a long study of it holds at once."""
    return n + n // 64 + (1 << 17) + (2 * f["inject_pairs"] * f["nth"] * 4000 if f["inject"] and n < 4e6 else 0)


def _simulation(f, n):
    dt, b0, qw, inject_q = _physics(f)
    d = P.make_desc(nr=f["nr"], nth=f["nth"], r_min=f["r_min"], r_max=f["r_max"], r_map=f["r_map"],
                    th_map=f["th_map"], dt=dt, n_filt=f["n_filt"], absorb_cells=f["absorb_cells"],
                    absorb_profile=f["absorb_profile"], vacuum=f["vacuum"], b0=b0, omega=f["omega"],
                    t_spin=f["t_spin"], inject=f["inject"], pairs_per_cell=f["inject_pairs"], f_inj=f["f_inj"],
                    precision=f["precision"], pusher=f["pusher"], q_over_m=1.0, sort_interval=f["sort_interval"],
                    inject_smooth=f["inject_smooth"], inject_q=inject_q, inject_seed=7,
                    capacity=_capacity(f, n))
    return P.Simulation(d, stream=torch.cuda.current_stream().cuda_stream)


def _table(T):
    u = np.linspace(0.0, max(40.0 * T + 10.0 * math.sqrt(T), 1.0), 1 << 14)
    pdf = u * u * np.exp(-(np.sqrt(1.0 + u * u) - 1.0) / T)
    cdf = np.concatenate([[0.0], np.cumsum(0.5 * (pdf[1:] + pdf[:-1]) * np.diff(u))])
    return cdf / cdf[-1], u


def _plasma(f, seed, total=None, chunk=1 << 22):
    """Co-located electron-positron pairs, `pairs` in every cell (or `total`
    particles spread over the cells), cell by cell, with isotropic
    Maxwell-Juettner momenta; chunks of FP64 device tensors.  For the FP32
    path the values are ones it holds exactly."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    cdf, u = (torch.tensor(a, device=DEV) for a in _table(f["T"]))
    qw = _physics(f)[2]
    ncell = f["nr"] * f["nth"]
    npair = ncell * f["pairs"] if total is None else total // 2
    rnd = lambda n: torch.rand(n, generator=g, device=DEV, dtype=torch.float32)  # noqa: E731
    for p0 in range(0, npair, chunk):
        m = min(chunk, npair - p0)
        k = torch.arange(p0, p0 + m, device=DEV)
        cell = k // f["pairs"] if total is None else k * ncell // npair
        # offsets are multiples of 2^-24 below 1: FP32 values
        x1 = ((cell // f["nth"]).double() + rnd(m).double()).repeat_interleave(2)
        x2 = ((cell % f["nth"]).double() + rnd(m).double()).repeat_interleave(2)
        U = torch.rand(2 * m, generator=g, device=DEV, dtype=torch.float64)
        q = torch.searchsorted(cdf, U).clamp_(1, len(cdf) - 1)
        mag = u[q - 1] + (U - cdf[q - 1]) / (cdf[q] - cdf[q - 1]).clamp_min(1e-300) * (u[q] - u[q - 1])
        ca = rnd(2 * m).double() * 2.0 - 1.0
        ph = rnd(2 * m).double() * (2.0 * math.pi)
        sa = (1.0 - ca * ca).clamp_min(0.0).sqrt()
        out = [x1, x2, mag * ca, mag * sa * torch.cos(ph), mag * sa * torch.sin(ph),
               torch.tensor([qw, -qw], device=DEV, dtype=torch.float64).repeat(m)]
        if f["precision"] == "fp32":
            out[2:] = [a.float().double() for a in out[2:]]
        yield out


def _members(case, seed):
    """The ensemble's members: uneven grids, particle counts and temperatures."""
    rng = np.random.default_rng(20140718)  # the sizes are the case's, the plasmas the seed's
    out = []
    for m in range(case["members"]):
        n = int(round(math.exp(math.log(case["n_lo"]) + rng.random() * math.log(case["n_hi"] / case["n_lo"]))))
        f = dict(MONOPOLE, nr=(64, 128, 256)[m % 3], nth=(64, 128, 256, 512)[(m // 3) % 4], r_max=10.0,
                 absorb_cells=8, T=0.05 + 0.95 * rng.random(), wp_dt=0.05, precision="fp32")
        f["pairs"] = max(1, n // (2 * f["nr"] * f["nth"]))
        out.append((f, n // 2 * 2, seed * 1000 + m))
    return out


def _count(f):
    return 2 * f["nr"] * f["nth"] * f["pairs"]


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["do"] == "ensemble":
        s.sims = []
        for f, n, sd in _members(case, seed):
            sim = _simulation(f, n)
            for a in _plasma(f, sd, total=n):
                sim.load(*a)
            s.sims.append(sim)
        return s
    f = s.f = _config(case)
    if case["do"] == "whole":
        parts = [torch.cat(a).cpu().pin_memory() for a in zip(*_plasma(f, seed))]
        s.host = parts
        return s
    s.sim = _simulation(f, _count(f))
    for a in _plasma(f, seed):
        s.sim.load(*a)
    if case["do"] == "diagnose":
        s.sim.step(case["steps"])
    torch.cuda.synchronize()
    return s


# ---- one pass -------------------------------------------------------------------
def _fields(sim, precision):
    """The plasma fields: a numpy array for a small grid, read on the device
    (as a GPU program does) for a large one."""
    if sim.nr * sim.nth <= 20000:
        out = sim.fields()
        return out.astype(np.float32) if precision == "fp32" else out
    n = C.c_int64()
    P.check(sim.L.pic_get_fields(sim.h, P.PIC_FIELDS_PLASMA, None, C.byref(n), P.PIC_MEM_DEVICE))
    out = torch.empty((6, sim.nr + 1, sim.nth + 1), device=DEV, dtype=torch.float64)
    P.check(sim.L.pic_get_fields(sim.h, P.PIC_FIELDS_PLASMA, C.c_void_p(out.data_ptr()), C.byref(n),
                                 P.PIC_MEM_DEVICE))
    return out.float() if precision == "fp32" else out


def run(state):
    case = state.case
    if case["do"] == "ensemble":
        P.ensemble_step(state.sims, case["steps"])
        return {"fields": [_fields(s, "fp32") for s in state.sims]}
    prec = state.f["precision"]
    if case["do"] == "whole":
        sim = _simulation(state.f, len(state.host[0]))
        sim.load(*state.host)
        sim.step(case["steps"])
        out = {"fields": _fields(sim, prec)}
        sim.close()
        return out
    sim = state.sim
    if case["do"] == "diagnose":
        m = sim.moments()
        n = C.c_int64()
        q = torch.empty((sim.nr + 2 * sim.g + 1, sim.nth + 1), device=DEV, dtype=torch.float64)
        P.check(sim.L.pic_get_charge(sim.h, 1, C.c_void_p(q.data_ptr()), C.byref(n), P.PIC_MEM_DEVICE))
        # (the Gauss residual and the total charge of a neutral plasma are
        # differences of rounding size: computed above, not compared)
        return {"live": m["live"], "deleted": m["deleted"],
                "energy": np.array([m["kinetic_energy"], m["field_energy"]], dtype=np.float32), "charge": q.float(),
                "luminosity": sim.luminosity().astype(np.float32)}
    sim.step(case["steps"])
    out = {"fields": _fields(sim, prec)}
    if prec == "fp64":
        out["particles"] = _padded(sim.particles(device=DEV), _capacity(state.f, _count(state.f)))
    return out


def _padded(parts, slots):
    """The live particles in buffers of a fixed size, as a program that keeps
    its own copies holds them."""
    out = {}
    for k, a in parts.items():
        out[k] = torch.zeros(slots, device=DEV, dtype=a.dtype)
        out[k][: len(a)] = a
    return out


def work(case):
    """Particle state read and written once a step (FP32: 28 B in, 24 B out;
    FP64: 48 B in, 40 B out), the grid's fields updated once a step, the
    fields read out.  Operations: a gather, push, move and deposit of about
    400 floating-point operations; the stencils' on the grid."""
    if case["do"] == "ensemble":
        fs = [(f, n) for f, n, _ in _members(case, 0)]
    else:
        f = _config(case)
        fs = [(f, _count(f))]
    b = w = 0.0
    for f, n in fs:
        nodes = (f["nr"] + 1) * (f["nth"] + 1)
        if case["do"] == "diagnose":
            b += n * 24 + nodes * (6 * 8 + 8 + 8)  # cell, offsets, momenta, charge; fields; charge out
            w += n * 60.0 + nodes * (40.0 + 24.0 * f["n_filt"])
            continue
        fp32 = f["precision"] == "fp32"
        out = 4 if fp32 else 8
        b += case["steps"] * (n * (52 if fp32 else 88) + nodes * (6 * 16 + 3 * 8 + (6 * 4 if fp32 else 0)))
        b += nodes * 6 * (8 + out) + (n * 48 if case["do"] == "whole" else 0)
        if not fp32:
            b += n * 2 * 56  # the particles read out
        w += case["steps"] * (n * 400.0 + nodes * (50.0 + 18.0 * f["n_filt"]))
    return {"bytes": b, "flops": w}


# ---- the method in plain FP64 torch operations ------------------------------------
SI, SJ = (1, 0, 0, 0, 1, 1), (0, 1, 0, 1, 0, 1)  # half-integer staggering of E_r E_th E_ph B_r B_th B_ph
ER, ETH, EPH, BR, BTH, BPH = range(6)


class _Exact:
    def __init__(self, f):
        self.f = f
        self.nr, self.nth, self.nf = f["nr"], f["nth"], f["n_filt"]
        self.g = self.nf + 2
        self.dt, self.b0, self.qw, self.inject_q = _physics(f)
        self.dxi = (math.log(f["r_max"] / f["r_min"]) if f["r_map"] == "log" else f["r_max"] - f["r_min"]) / f["nr"]
        # fields with one ghost row and column on each side: [i + 1][j + 1]
        self.F6 = [self._zeros(self.nr + 3, self.nth + 3) for _ in range(6)]
        self.step_no = 0
        self.deleted = 0
        self.next_id = 0
        t = lambda a: torch.tensor(a, device=DEV, dtype=torch.float64)  # noqa: E731
        i = np.arange(-1.0, self.nr + 2.0)  # i + 1 indexed
        self.rn, self.rh = t(_fr(f, i))[:, None], t(_fr(f, i + 0.5))[:, None]
        j = np.arange(self.nth + 1.0)
        self.th, self.tb = _fth(f, j), _fth(f, j[:-1] + 0.5)
        ctb = np.concatenate([[1.0], np.cos(self.tb), [-1.0]])  # cos tb_{j-1} at [j], caps at the axis
        self.dcos_tb = t(ctb[:-1] - ctb[1:])[None]               # dual cell of node j
        self.stb = t(np.sin(self.tb))[None]
        self.ctb = t(np.cos(self.tb))[None]
        self.st, self.ct = t(np.sin(self.th))[None], t(np.cos(self.th))[None]
        self.dcos = t(np.cos(self.th[:-1]) - np.cos(self.th[1:]))[None]
        self.dth = t(np.diff(self.th))[None]
        self.dtb = t(np.diff(self.tb))[None]
        self.parts = [torch.empty(0, device=DEV, dtype=torch.float64) for _ in range(6)]
        self.ids = torch.empty(0, device=DEV, dtype=torch.int64)

    @staticmethod
    def _zeros(*s):
        return torch.zeros(s, device=DEV, dtype=torch.float64)

    def load(self, chunks):
        self.parts = [torch.cat(a) for a in zip(*chunks)]
        n = len(self.parts[0])
        self.ids = torch.arange(n, device=DEV)
        self.next_id = n

    def omega(self, t):
        f = self.f
        return f["omega"] * (t / f["t_spin"]) if f["t_spin"] > 0 and t < f["t_spin"] else f["omega"]

    def vacuum(self, r, st, ct, inside, t):
        """The analytic field (E, B) in spherical components; `inside`: a mask
        or truth value for points inside the star."""
        b0, r0, W, kind = self.b0, self.f["r_min"], self.omega(t), self.f["vacuum"]
        z = torch.zeros_like(r * st)
        pick = lambda a, b: torch.where(inside, a, b) if isinstance(inside, torch.Tensor) else (a if inside else b)  # noqa: E731
        q2 = (r0 / r) ** 2
        if kind == "monopole":
            return [z, z, z], [b0 * q2 + z, z, z]
        if kind == "monopole_rotator":
            a = b0 * q2 * (r0 * r0 / r) * W
            return [pick(z, -2.0 * a * ct), pick(-b0 * r0 * r0 / r * W * st, -a * st), z], [b0 * q2 + z, z, z]
        mu = b0 * r0 ** 3  # dipole_rotator
        a = mu * W * q2 / (r * r)
        E = [pick(mu * W * st * st / (r * r), -a * (3.0 * ct * ct - 1.0)),
             pick(-2.0 * mu * W * st * ct / (r * r), -2.0 * a * st * ct), z]
        return E, [2.0 * mu * ct / r ** 3, mu * st / r ** 3, z]

    def ghosts(self):
        n = self.nth + 1  # column index of j = nth
        for k, s in ((ETH, -1.0), (BR, 1.0), (BPH, -1.0)):
            a = self.F6[k]
            a[1:-1, 0] = s * a[1:-1, 1]
            a[1:-1, n] = s * a[1:-1, n - 1]

    def gather(self, k, x1, x2):
        p1, p2 = x1 - 0.5 * SI[k], x2 - 0.5 * SJ[k]
        a, b = torch.floor(p1), torch.floor(p2)
        w1, w2 = p1 - a, p2 - b
        o = (a.long() + 1) * (self.nth + 3) + b.long() + 1
        F = self.F6[k].view(-1)
        ld = self.nth + 3
        return ((1 - w1) * (1 - w2) * F[o] + w1 * (1 - w2) * F[o + ld] + (1 - w1) * w2 * F[o + 1]
                + w1 * w2 * F[(o + ld + 1).clamp_max(F.numel() - 1)])

    def push(self, qmdt, E, B, u):
        cross = lambda a, b: [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]  # noqa: E731
        dot = lambda a, b: a[0] * b[0] + a[1] * b[1] + a[2] * b[2]  # noqa: E731
        h = 0.5 * qmdt
        if self.f["pusher"] == "boris":
            m = [u[k] + h * E[k] for k in range(3)]
            ig = 1.0 / torch.sqrt(1.0 + dot(m, m))
            t = [h * B[k] * ig for k in range(3)]
            c = cross(m, t)
            p = [m[k] + c[k] for k in range(3)]
            s = 2.0 / (1.0 + dot(t, t))
            c = cross(p, t)
            return [m[k] + s * c[k] + h * E[k] for k in range(3)]
        ig = 1.0 / torch.sqrt(1.0 + dot(u, u))
        tau = [h * B[k] for k in range(3)]
        c = cross([a * ig for a in u], tau)
        a = [u[k] + qmdt * E[k] + c[k] for k in range(3)]
        t2, us = dot(tau, tau), dot(a, tau)
        sg = 1.0 + dot(a, a) - t2
        g = torch.sqrt(0.5 * (sg + torch.sqrt(sg * sg + 4.0 * (t2 + us * us))))
        t = [x / g for x in tau]
        s = 1.0 / (1.0 + dot(t, t))
        at = dot(a, t)
        c = cross(a, t)
        return [s * (a[k] + at * t[k] + c[k]) for k in range(3)]

    def fluxes(self):
        return [self._zeros((self.nr + 2 * self.g + 3) * (self.nth + 3)) for _ in range(3)]

    def node(self, i, j):  # flat index of node (i, j) in a flux array
        return (i + self.g + 1) * (self.nth + 3) + j + 1

    def segment(self, D, q, ic, jc, p, e):
        d1, d2 = e[0] - p[0], e[1] - p[1]
        m1, m2 = 0.5 * (p[0] + e[0]) - ic, 0.5 * (p[1] + e[1]) - jc
        o = self.node(ic, jc)
        D[0].index_add_(0, o, q * d1 * (1.0 - m2))
        D[0].index_add_(0, o + 1, q * d1 * m2)
        D[1].index_add_(0, o, q * d2 * (1.0 - m1))
        D[1].index_add_(0, o + (self.nth + 3), q * d2 * m1)

    def particles(self, part, D, t):
        """One step of some particles: their new state, deposit into D."""
        x1, x2, ur, ut, up, q = part
        f, nr, nth = self.f, self.nr, self.nth
        r = f["r_min"] * torch.exp(x1 * self.dxi) if f["r_map"] == "log" else f["r_min"] + x1 * self.dxi
        th = torch.arccos(1.0 - 2.0 * x2 / nth) if f["th_map"] == "equal_area" else math.pi / nth * x2
        st, ct = torch.sin(th), torch.cos(th)
        inside, free = x1 < 0.0, x1 >= nr
        E, B = self.vacuum(r, st, ct, inside, t)
        off = inside | free
        g1, g2 = torch.where(off, 0.5, x1), x2
        for k in range(3):
            E[k] = E[k] + torch.where(off, 0.0, self.gather(k, g1, g2))
            B[k] = B[k] + torch.where(off, 0.0, self.gather(3 + k, g1, g2))
        u = [ur, ut, up]
        v = self.push(torch.sign(q) * self.dt, E, B, u)
        u = [torch.where(free, a, b) for a, b in zip(u, v)]
        del E, B, v
        # straight 3-D move in Cartesian components at phi = 0, then back
        ux, uy, uz = u[0] * st + u[1] * ct, u[2], u[0] * ct - u[1] * st
        s = self.dt / torch.sqrt(1.0 + ux * ux + uy * uy + uz * uz)
        X, Y, Z = r * st + ux * s, uy * s, r * ct + uz * s
        R = torch.hypot(X, Y)
        rn, thn, phi = torch.hypot(R, Z), torch.atan2(R, Z), torch.atan2(Y, X)
        cp, sp = torch.where(R > 0, X / R, 1.0), torch.where(R > 0, Y / R, 0.0)
        ux, uy = cp * ux + sp * uy, cp * uy - sp * ux
        stn, ctn = R / rn, Z / rn
        n1 = torch.log(rn / f["r_min"]) / self.dxi if f["r_map"] == "log" else (rn - f["r_min"]) / self.dxi
        n2 = 0.5 * nth * (1.0 - torch.cos(thn)) if f["th_map"] == "equal_area" else thn * (nth / math.pi)
        n2 = n2.clamp(0.0, nth)
        new = [n1, n2, ux * stn + uz * ctn, ux * ctn - uz * stn, uy, q]
        # the path in grid coordinates, split where it crosses grid lines
        fl = lambda a: torch.floor(a).long()  # noqa: E731
        ia, ib = fl(x1), fl(n1)
        ja, jb = fl(x2).clamp(0, nth - 1), fl(n2).clamp(0, nth - 1)
        cx, cy = ia != ib, ja != jb
        X, Y = torch.maximum(ia, ib).double(), torch.maximum(ja, jb).double()
        sx = torch.where(cx, (X - x1) / (n1 - x1), 2.0)
        sy = torch.where(cy, (Y - x2) / (n2 - x2), 2.0)
        P0, ic, jc = (x1, x2), ia, ja
        for _ in range(2):
            xf = sx <= sy
            sn = torch.where(xf, sx, sy)
            hit = sn <= 1.0
            jd, idb = jc.double(), ic.double()
            a2 = torch.minimum(torch.maximum(x2 + sn * (n2 - x2), jd), jd + 1.0)
            a1 = torch.minimum(torch.maximum(x1 + sn * (n1 - x1), idb), idb + 1.0)
            Q = (torch.where(hit, torch.where(xf, X, a1), n1), torch.where(hit, torch.where(xf, a2, Y), n2))
            self.segment(D, q, ic, jc, P0, Q)
            P0 = Q
            ic, jc = torch.where(hit & xf, ib, ic), torch.where(hit & ~xf, jb, jc)
            sx, sy = torch.where(xf, 2.0, sx), torch.where(xf, sy, 2.0)
        self.segment(D, q, ic, jc, P0, (n1, n2))
        m1, m2 = 0.5 * (x1 + n1), 0.5 * (x2 + n2)
        fi, fj = torch.floor(m1), torch.floor(m2)
        w1, w2, w = m1 - fi, m2 - fj, q * phi * (0.5 / math.pi)
        o, ld = self.node(fi.long(), fj.long()), nth + 3
        D[2].index_add_(0, o, w * (1 - w1) * (1 - w2))
        D[2].index_add_(0, o + ld, w * w1 * (1 - w2))
        D[2].index_add_(0, o + 1, w * (1 - w1) * w2)
        D[2].index_add_(0, o + ld + 1, w * w1 * w2)
        return new, (ib >= -(self.nf + 1)) & (ib < nr + self.nf + 1)

    def filtered(self, a, half):
        """The 1-2-1 passes with the polar fold on rows -g..nr+g, nodes 0..nth
        (the half-integer component: 0..nth-1)."""
        a = a.view(self.nr + 2 * self.g + 3, self.nth + 3)[1:-1, 1: (-2 if half else -1)]
        for _ in range(self.nf):
            n = a.shape[1]
            vm, v0, vp = torch.full((n,), 0.25), torch.full((n,), 0.5), torch.full((n,), 0.25)
            vm[0], vp[-1] = 0.0, 0.0
            if half:
                v0[0] -= 0.25
                v0[-1] -= 0.25
            else:
                vm[1], vp[-2] = 0.5, 0.5
            vm, v0, vp = (v.double().to(DEV) for v in (vm, v0, vp))
            b = v0 * a
            b[:, 1:] += vm[1:] * a[:, :-1]
            b[:, :-1] += vp[:-1] * a[:, 1:]
            a = 0.5 * b
            a[1:] += 0.25 * b[:-1]
            a[:-1] += 0.25 * b[1:]
        return a

    def b_half(self):
        nr, nth, h = self.nr, self.nth, 0.5 * self.dt
        Er, Et, Ep, Br, Bt, Bp = self.F6
        N = lambda a, i, j, di=0, dj=0: a[1 + di: 1 + di + i, 1 + dj: 1 + dj + j]  # noqa: E731
        r, r1 = self.rn[1: 1 + nr], self.rn[2: 2 + nr]
        A = h * 2.0 / (r1 * r1 - r * r)
        N(Br, nr + 1, nth).add_(h / self.rn[1: 2 + nr] * (N(Ep, nr + 1, nth) * self.st[:, :-1]
                                - N(Ep, nr + 1, nth, dj=1) * self.st[:, 1:]) / self.dcos)
        Bt[1: 1 + nr, 2: 1 + nth] += A * (r1 * Ep[2: 2 + nr, 2: 1 + nth] - r * Ep[1: 1 + nr, 2: 1 + nth])
        N(Bp, nr, nth).add_(A * (r * N(Et, nr, nth) - r1 * N(Et, nr, nth, di=1)
                            - (r1 - r) / self.dth * (N(Er, nr, nth) - N(Er, nr, nth, dj=1))))

    def e_full(self, F):
        nr, nth, dt, g = self.nr, self.nth, self.dt, self.g
        Er, Et, Ep, Br, Bt, Bp = self.F6
        pi2 = 2.0 * math.pi
        rh, rm = self.rh[2: 1 + nr], self.rh[1: nr]          # rb_i, rb_{i-1} for i = 1..nr-1
        A = 2.0 / (rh * rh - rm * rm)
        rb = self.rh[1: 1 + nr]                               # rb_i, i = 0..nr-1
        sB = torch.zeros(nr, nth + 2, device=DEV, dtype=torch.float64)
        sB[:, 1:-1] = Bp[1: 1 + nr, 1: 1 + nth] * self.stb    # sin tb_j B_ph, zero beyond the poles
        Er[1: 1 + nr, 1: 2 + nth] += (dt / rb * (sB[:, 1:] - sB[:, :-1]) / self.dcos_tb
                                      - F[0][g: g + nr, : nth + 1] / (pi2 * rb * rb * self.dcos_tb))
        Et[2: 1 + nr, 1: 1 + nth] += (A * dt * (rm * Bp[1: nr, 1: 1 + nth] - rh * Bp[2: 1 + nr, 1: 1 + nth])
                                      - F[1][g + 1: g + nr, :nth] * A / (pi2 * self.stb))
        Ep[2: 1 + nr, 2: 1 + nth] += (A * dt * (rh * Bt[2: 1 + nr, 2: 1 + nth] - rm * Bt[1: nr, 2: 1 + nth]
                                      - (rh - rm) / self.dtb * (Br[2: 1 + nr, 2: 1 + nth] - Br[2: 1 + nr, 1: nth]))
                                      - F[2][g + 1: g + nr, 1: nth] * A / self.dtb)

    def lossy(self):
        f, L = self.f, self.f["absorb_cells"]
        rho = torch.arange(-1.0, self.nr + 2.0, device=DEV, dtype=torch.float64)[:, None]
        for k in range(6):
            u = ((rho + 0.5 * SI[k]) - (self.nr - L)).clamp_min(0.0) / L
            s = 3.0 / L * u * u if f["absorb_profile"] == "quadratic" else 2.0 / L * u
            self.F6[k] *= 1.0 - s

    def inject(self):
        f, nth, npp = self.f, self.nth, self.f["inject_pairs"]
        t = self.step_no * self.dt
        rb0 = self.rh[1]
        out, _ = self.vacuum(rb0, self.st[0], self.ct[0], False, t)
        ins, _ = self.vacuum(torch.full_like(rb0, f["r_min"]), self.st[0], self.ct[0], True, t)
        e = self.F6[ER][1, 1: 2 + nth] + out[0] - ins[0]
        sg = 0.5 * (e[:-1] + e[1:])
        for _ in range(f["inject_smooth"]):
            p = torch.cat([sg[:1], sg, sg[-1:]])
            sg = 0.25 * (p[:-2] + 2.0 * sg + p[2:])
        sg = sg.cpu().numpy()
        on = np.abs(sg) > 1e-12 * np.abs(sg).max()
        dA = 2.0 * math.pi * f["r_min"] ** 2 * self.dcos[0].cpu().numpy()
        w = f["f_inj"] * np.abs(sg) * dA
        if f["inject"] == 2:
            x = w / self.inject_q
            with np.errstate(over="ignore"):
                k = np.uint64(self.step_no) * np.uint64(nth) + np.arange(nth, dtype=np.uint64) + np.uint64(1)
                z = np.uint64(7) + k * np.uint64(0x9E3779B97F4A7C15)
                z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
                z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
                z = z ^ (z >> np.uint64(31))
            m = np.floor(x) + ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 < x - np.floor(x))
            m = np.where(on & (x > 0), np.minimum(m, npp), 0).astype(int)
            w = np.full(nth, self.inject_q)
        else:
            m = np.where(on & (w > 0), npp, 0)
            w = w / npp
        jj, kk, ss = np.meshgrid(np.arange(nth), np.arange(npp), np.arange(2), indexing="ij")
        sel = (kk < m[:, None, None]).ravel()
        slot = np.arange(sel.size)[sel]
        jj, kk, ss = jj.ravel()[sel], kk.ravel()[sel], ss.ravel()[sel]
        new = [np.full(len(jj), 0.5), jj + (kk + 0.5) / m[jj], np.zeros(len(jj)), np.zeros(len(jj)),
               np.zeros(len(jj)), np.where(ss == 0, w[jj], -w[jj])]
        self.parts = [torch.cat([a, torch.tensor(b, device=DEV, dtype=torch.float64)])
                      for a, b in zip(self.parts, new)]
        self.ids = torch.cat([self.ids, torch.tensor(self.next_id + slot, device=DEV)])
        self.next_id += sel.size

    def step(self, chunk=1 << 22):
        t = self.step_no * self.dt
        D = self.fluxes()
        self.ghosts()
        keep = []
        for a in range(0, len(self.ids), chunk):
            b = min(a + chunk, len(self.ids))
            new, alive = self.particles([p[a:b] for p in self.parts], D, t)
            for p, q in zip(self.parts, new):
                p[a:b] = q
            keep.append(alive)
        if keep:
            keep = torch.cat(keep)
            if not bool(keep.all()):
                self.deleted += int((~keep).sum())
                self.parts = [p[keep] for p in self.parts]
                self.ids = self.ids[keep]
        F = [self.filtered(D[0], False), self.filtered(D[1], True), self.filtered(D[2], False)]
        self.b_half()
        self.e_full(F)
        self.b_half()
        self.lossy()
        self.step_no += 1
        if self.f["inject"]:
            self.inject()

    def fields(self):
        out = self._zeros(6, self.nr + 1, self.nth + 1)
        for k in range(6):
            n, m = self.nr + 1 - SI[k], self.nth + 1 - SJ[k]
            out[k, :n, :m] = self.F6[k][1: 1 + n, 1: 1 + m]
        return out

    def charge(self):
        Q = self.fluxes()[0]
        x1, x2, q = self.parts[0], self.parts[1], self.parts[5]
        for a in range(0, len(q), 1 << 24):
            y1, y2, w = x1[a: a + (1 << 24)], x2[a: a + (1 << 24)], q[a: a + (1 << 24)]
            fi, fj = torch.floor(y1), torch.floor(y2)
            w1, w2 = y1 - fi, y2 - fj
            o, ld = self.node(fi.long(), fj.long()), self.nth + 3
            Q.index_add_(0, o, w * (1 - w1) * (1 - w2))
            Q.index_add_(0, o + ld, w * w1 * (1 - w2))
            Q.index_add_(0, o + 1, w * (1 - w1) * w2)
            Q.index_add_(0, o + ld + 1, w * w1 * w2)
        return self.filtered(Q, False)

    def energies(self):
        kin = 0.0
        for a in range(0, len(self.ids), 1 << 24):
            ur, ut, up, q = (p[a: a + (1 << 24)] for p in self.parts[2:])
            u2 = ur * ur + ut * ut + up * up
            kin += float((q.abs() * (u2 / (1.0 + torch.sqrt(1.0 + u2)))).sum())
        f = self.f
        i, j = np.arange(self.nr + 1.0), np.arange(self.nth + 1.0)
        e = 0.0
        for k in range(6):
            lo, hi = (i, np.minimum(i + 1, self.nr)) if SI[k] else (np.maximum(i - 0.5, 0), np.minimum(i + 0.5, self.nr))
            vr = 2 * math.pi / 3 * (_fr(f, hi) ** 3 - _fr(f, lo) ** 3)
            lo, hi = (j, np.minimum(j + 1, self.nth)) if SJ[k] else (np.maximum(j - 0.5, 0), np.minimum(j + 0.5, self.nth))
            vt = np.cos(_fth(f, lo)) - np.cos(_fth(f, hi))
            V = torch.tensor(vr[:, None] * vt[None], device=DEV)
            e += 0.5 * float((self.F6[k][1:-1, 1:-1] ** 2 * V).sum())
        return np.array([kin, e])

    def luminosity(self):
        nr, nth = self.nr, self.nth
        t = self.step_no * self.dt
        r = self.rn[2: 1 + nr]
        E, B = self.vacuum(r, self.stb, self.ctb, False, t)
        I = lambda a, di, dj: a[2 + di: 1 + nr + di, 1 + dj: 1 + nth + dj]  # noqa: E731, E741
        _, Et, Ep, _, Bt, Bp = self.F6
        et = I(Et, 0, 0) + E[1]
        bp = 0.5 * (I(Bp, -1, 0) + I(Bp, 0, 0)) + B[2]
        ep = 0.5 * (I(Ep, 0, 0) + I(Ep, 0, 1)) + E[2]
        bt = 0.25 * (I(Bt, -1, 0) + I(Bt, 0, 0) + I(Bt, -1, 1) + I(Bt, 0, 1)) + B[1]
        L = np.zeros(nr + 1)
        L[1:nr] = ((et * bp - ep * bt) * (2.0 * math.pi * r * r) * self.dcos).sum(1).cpu().numpy()
        return L


def exact(case, seed):
    if case["do"] == "ensemble":
        out = []
        for f, n, sd in _members(case, seed):
            x = _Exact(f)
            x.load(list(_plasma(f, sd, total=n)))
            for _ in range(case["steps"]):
                x.step()
            out.append(x.fields())
        return {"fields": out}
    f = _config(case)
    if _count(f) * case["steps"] > 2.2e9:
        return None
    x = _Exact(f)
    x.load(list(_plasma(f, seed)))
    for _ in range(case["steps"]):
        x.step()
    if case["do"] == "diagnose":
        return {"live": None, "deleted": None, "energy": x.energies(), "charge": x.charge(),
                "luminosity": x.luminosity()}
    out = {"fields": x.fields()}
    if f["precision"] == "fp64":
        out["particles"] = dict(_padded(dict(zip(("x1", "x2", "ur", "uth", "uph", "qw"), x.parts)),
                                        _capacity(f, _count(f))), id=None)
    return out
