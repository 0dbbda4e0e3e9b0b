"""Workloads of the Lagrangian-mean library for timing and for comparing results.

A case is a dict of plain values; `prepare` makes its inputs and handles on
the GPU, `run` does one pass through the public binding as a user's program
does, `work` counts what a pass cannot do without, and `exact` computes the
same outputs in FP64 with plain torch (2D real FFTs over the full grid).

Kinds of case:
  interval  one averaging interval (initial condition in, n steps, means out)
            of one handle, or of several handles stepped as one batch
  steps     dynamics only: n steps, then the fields
  sl        a semi-Lagrangian Strategy-1 interval
  remap     Strategy-1 means onto the mean-position grid

FP32 runs return their results as float32 (their means leave the library as
FP64 arrays that carry FP32 accuracy).
"""
from __future__ import annotations

import math

import torch

import paper_2208_02682_gb300 as lm

DEV = "cuda"
SCALARS = ("zeta", "h", "u", "v", "q")
STAGES = {"rk4": 4, "heun": 2, "euler": 1}


# ---------------------------------------------------------------------------
# Cases

def listed():
    return [
        # a user who steps a small run and looks at its fields every few
        # steps: launches and host latency
        dict(name="steps-64-f32", kind="steps", N=64, prec="f32", n=8),
        # the test-size workload (64^2, FP64, Strategy 1), one wave period
        dict(name="s1-64-f64", kind="interval", N=64, prec="f64", strategy="1", fields="zeta,h,u,v", n=305),
        # the benchmark: both strategies of the 256^2 workload as one batch,
        # FP32, one wave period
        dict(name="s1s2-256-f32", kind="interval", N=256, prec="f32", strategy="1,2", fields="zeta,h,u,v", n=305),
        # the same workload in FP64, a single run
        dict(name="s1-256-f64", kind="interval", N=256, prec="f64", strategy="1", fields="zeta,h,u,v", n=64),
        # Strategy 2 with the potential vorticity averaged
        dict(name="s2q-512-f32", kind="interval", N=512, prec="f32", strategy="2", fields="zeta,h,u,v,q", n=64),
        # the precision workload in both precisions
        dict(name="s1-1024-f32", kind="interval", N=1024, prec="f32", strategy="1", fields="zeta,h,u,v", n=48),
        dict(name="s1-1024-f64", kind="interval", N=1024, prec="f64", strategy="1", fields="zeta,h,u,v", n=8),
        # the largest grid
        dict(name="s1-2048-f32", kind="interval", N=2048, prec="f32", strategy="1", fields="zeta,h,u,v", n=16),
        # an ensemble of different grid sizes stepped as one batch
        dict(name="ensemble-f32", kind="interval", N="128,256,512,256,128,512,256,128,512,128,256,512", prec="f32",
             strategy="1", fields="zeta,h,u,v", n=32),
        # the paper's vortex merger (two-dimensional Euler flow, Heun)
        dict(name="merger-128-f64", kind="interval", N=128, prec="f64", strategy="1", fields="zeta", n=400,
             model="euler2d", stepper="heun", eulerian=False, pos=False),
        # the semi-Lagrangian variant (FP64 means on FP32 dynamics)
        dict(name="sl-256-f32", kind="sl", N=256, prec="f32", fields="zeta,h,u,v", scheme="trapezoid", interp="cubic",
             n=64),
        # Strategy-1 results onto the mean-position grid
        dict(name="remap-1024", kind="remap", N=1024, fields="zeta,h,u,v", iters=20),
    ]


def _subset(rng, names):
    s = [f for f in names if rng.random() < 0.7]
    return ",".join(s or [rng.choice(list(names))])


def draw(rng):
    kind = rng.choices(("interval", "batch", "steps", "sl", "remap", "merger"), (8, 2, 2, 2, 1, 1))[0]
    if kind == "remap":
        return dict(kind="remap", N=2 ** rng.randint(5, 11), fields=_subset(rng, SCALARS[:4]), iters=rng.randint(8, 30))
    if kind == "merger":
        return dict(kind="interval", N=2 ** rng.randint(5, 8), prec=rng.choice(("f32", "f64")), strategy="1",
                    fields=_subset(rng, ("zeta", "u", "v")), n=rng.randint(20, 200), model="euler2d",
                    stepper=rng.choice(("heun", "rk4")), eulerian=rng.random() < 0.5, pos=rng.random() < 0.5)
    prec = rng.choice(("f32", "f64"))
    logn = rng.randint(4, 11 if prec == "f32" else 10)
    # steps: about the same total work for every size, at most one wave period
    most = max(3, min(305, (1 << (24 if prec == "f32" else 22)) >> (2 * logn)))
    n = max(1, int(round(math.exp(rng.uniform(0.0, math.log(most))))))
    if kind == "steps":
        return dict(kind="steps", N=2 ** logn, prec=prec, n=n, stepper=rng.choice(("rk4", "rk4", "heun", "euler")))
    if kind == "sl":
        return dict(kind="sl", N=2 ** min(logn, 9), prec=prec, fields=_subset(rng, SCALARS), n=min(n, 64),
                    scheme=rng.choice(("euler", "trapezoid")), interp=rng.choice(("linear", "cubic")))
    if kind == "batch":
        sizes = [2 ** rng.randint(6, 9) for _ in range(rng.randint(2, 6))]
        strat = ",".join(rng.choice("12") for _ in sizes)
        return dict(kind="interval", N=",".join(map(str, sizes)), prec=prec, strategy=strat,
                    fields=_subset(rng, SCALARS), n=rng.randint(2, 24), eulerian=rng.random() < 0.7)
    return dict(kind="interval", N=2 ** logn, prec=prec, strategy=rng.choice("12"), fields=_subset(rng, SCALARS), n=n,
                stepper=rng.choice(("rk4", "rk4", "rk4", "heun")), visc=rng.choice(("hyper8", "hyper8", "laplace")),
                eulerian=rng.random() < 0.7, pos=rng.random() < 0.8)


def _runs(case):
    """(N, strategy) of each handle of an interval."""
    N, s = str(case["N"]).split(","), str(case["strategy"]).split(",")
    k = max(len(N), len(s))
    return [(int(N[i % len(N)]), int(s[i % len(s)])) for i in range(k)]


def _fields(case):
    return tuple(f for f in SCALARS if f in case["fields"].split(","))


def _model(case):
    return case.get("model", "sw")


def _dt(N, case):
    return 5e-3 if N <= 1024 or case["kind"] == "remap" else 2.07e-3


def _nu(N, case):
    if _model(case) == "euler2d":
        return 0.0
    if case.get("visc", "hyper8") == "laplace":
        return 1e-4
    return 10.0 / float((N - 1) // 3) ** 8


def _keys(case, strategy):
    """Output names of an interval, in the library's order."""
    keys = list(_fields(case))
    if strategy == 2 or case.get("pos", True):
        keys += ["pos_x", "pos_y"]
    if case.get("eulerian", True) and case["kind"] == "interval":
        keys += ["e_" + f for f in _fields(case)]
    return keys


# ---------------------------------------------------------------------------
# Inputs

def _grid(N):
    x = torch.arange(N, dtype=torch.float64, device=DEV) * (2.0 * math.pi / N)
    return x[None, :].expand(N, N), x[:, None].expand(N, N)


def _wavenumbers(N):
    kx = torch.arange(N // 2 + 1, dtype=torch.float64, device=DEV)[None, :]
    ky = torch.fft.fftfreq(N, d=1.0 / N, dtype=torch.float64, device=DEV)[:, None]
    return kx, ky


def _flow(N, gen, ro=0.1, ratio=1.0):
    """Balanced turbulence of Rossby number `ro` (spectral peak 6, or lower on
    the smallest grids) plus Poincare waves of `ratio` times its energy:
    (3, N, N) fields u, v, h, f0 = c2 = 1."""
    kx, ky = _wavenumbers(N)
    K = (N - 1) // 3
    k2 = kx * kx + ky * ky
    kk = torch.sqrt(k2).clamp_min(1.0)
    box = (kx <= K) & (ky.abs() <= K) & (k2 > 0)
    peak = min(6.0, K / 2.0)

    def noise():
        return torch.fft.rfft2(torch.randn(N, N, dtype=torch.float64, device=DEV, generator=gen)) / N

    def phys(F):
        return torch.fft.irfft2(F, s=(N, N))

    psi = noise() * torch.where(box, torch.sqrt(kk * torch.exp(-2.0 * (kk / peak) ** 2)), 0.0)
    psi = psi * (ro / phys(-k2 * psi).square().mean().sqrt())
    bal = torch.stack([phys(-1j * ky * psi), phys(1j * kx * psi), phys(psi)])
    # linear waves: eigenvectors (i w k + f0 k_perp terms) of the linearised equations
    ring = box & (kk >= min(4.0, K / 2.0)) & (kk <= min(6.0, K - 1.0))
    om = torch.sqrt(1.0 + k2)
    eta = noise() * torch.where(ring, 1.0, 0.0)
    k2s = k2.clamp_min(1.0)
    wav = torch.stack([phys((kx * om + 1j * ky) * eta / k2s), phys((ky * om - 1j * kx) * eta / k2s), phys(eta)])
    wav = wav * torch.sqrt(ratio * bal.square().sum() / wav.square().sum())
    uvh = bal + wav
    uvh[2] += 1.0
    return uvh.contiguous()


def _vortices(N, gen):
    """Two like-signed Gaussian vortices that merge, their places varied."""
    X, Y = _grid(N)
    d = 0.1 * torch.rand(4, dtype=torch.float64, device=DEV, generator=gen)
    z = (torch.exp(-(X - math.pi + 0.1 + d[0]) ** 2 - (Y - math.pi + math.pi / 3 + d[1]) ** 2)
         + torch.exp(-(X - math.pi - 0.1 + d[2]) ** 2 - (Y - math.pi - math.pi / 3 + d[3]) ** 2))
    return torch.stack([torch.zeros_like(z), torch.zeros_like(z), z]).contiguous()


def _initial(case, N, gen):
    if _model(case) == "euler2d":
        return _vortices(N, gen)
    return _flow(N, gen, 0.05 if N >= 1024 else 0.1, 2.0 if N >= 1024 else 1.0)


def _initials(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    sizes = [N for N, _ in _runs(case)] if case["kind"] == "interval" else [int(case["N"])]
    return [_initial(case, N, gen) for N in sizes]


def _remap_inputs(case, seed):
    """Mean positions of a smooth invertible map and averaged fields."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    N = int(case["N"])
    X, Y = _grid(N)
    a, b = _flow(N, gen), _flow(N, gen)
    # displacements of a few cells, |grad d| well below 1
    pos = torch.stack([X - 0.6 * a[0], Y - 0.6 * a[1]])
    src = {"zeta": b[0] - b[1], "h": b[2], "u": b[0], "v": b[1]}
    return pos, {k: src[k].contiguous() for k in _fields(case)}


class _State:
    """Handles and buffers of a case; frees the handles with itself."""

    def __init__(self, case):
        self.case = case
        self.handles, self.batch = [], None

    def __del__(self):
        if self.batch is not None:
            lm.sw_batch_destroy(self.batch)
        for h in self.handles:
            lm.sw_destroy(h)


def prepare(case, seed):
    lm.build()
    s = _State(case)
    if case["kind"] == "remap":
        s.pos, s.src = _remap_inputs(case, seed)
        return s
    s.ics = _initials(case, seed)
    for ic in s.ics:
        N = ic.shape[-1]
        p = lm.make_params(N, _dt(N, case), precision=case["prec"], model=_model(case), nu8=_nu(N, case),
                           stepper=case.get("stepper", "rk4"), visc=case.get("visc", "hyper8"))
        s.handles.append(lm.sw_create(p, ic))
    if case["kind"] == "steps":
        s.out = [torch.empty_like(s.ics[0])]
        return s
    if case["kind"] == "sl":
        s.keys = [_keys(case, 1)]
        s.p = lm.make_sl_params(_fields(case), pos=True, scheme=case["scheme"], interp=case["interp"],
                                n_steps=case["n"])
    else:
        runs = _runs(case)
        s.keys = [_keys(case, st) for _, st in runs]
        s.p = [lm.make_lm_params(st, _fields(case), pos=case.get("pos", True),
                                 eulerian=case.get("eulerian", True), n_steps=case["n"]) for _, st in runs]
        if len(s.handles) > 1:
            s.batch = lm.sw_batch_create(s.handles)
    s.out = [torch.empty((len(k), ic.shape[-1], ic.shape[-1]), dtype=torch.float64, device=DEV)
             for k, ic in zip(s.keys, s.ics)]
    s.views = _named(s.keys, s.out)
    if case["prec"] == "f32":
        s.out32 = [torch.empty_like(o, dtype=torch.float32) for o in s.out]
        s.views32 = _named(s.keys, s.out32)
    return s


def _named(keys, stacks):
    """One dict of fields by name per run, views of the run's stack."""
    return [dict(zip(k, o.unbind(0))) for k, o in zip(keys, stacks)]


# ---------------------------------------------------------------------------
# One pass

def run(s):
    """The results by name, one dict per run (a stack of fields per run for
    larger ensembles)."""
    case = s.case
    if case["kind"] == "remap":
        return lm.lmean_remap(s.pos[0], s.pos[1], s.src, iters=case["iters"])
    for h, ic in zip(s.handles, s.ics):
        lm.sw_set_fields(h, ic)
    if case["kind"] == "steps":
        lm.sw_step(s.handles[0], case["n"])
        lm.sw_get_fields(s.handles[0], s.out[0])
        return s.out[0].float() if case["prec"] == "f32" else s.out[0]
    if case["kind"] == "sl":
        i = lm.sw_sl_create(s.handles[0], s.p)
        lm.sw_sl_step(i, case["n"])
        lm.sw_sl_end(i, s.views[0])
    else:
        for h, p in zip(s.handles, s.p):
            lm.lmean_begin(h, p)
        if s.batch is not None:
            lm.sw_batch_step(s.batch, case["n"])
        else:
            lm.lmean_step(s.handles[0], case["n"])
        for h, v in zip(s.handles, s.views):
            lm.lmean_end(h, v)
    if case["prec"] == "f32":
        for o32, o in zip(s.out32, s.out):
            o32.copy_(o)
        return s.views32 if len(s.keys) <= 4 else s.out32
    return s.views if len(s.keys) <= 4 else s.out


# ---------------------------------------------------------------------------
# Work of a pass: the initial condition read and the results written once
# and, every step, the evolved spectral state (2/3 box) read and written once;
# conventional flops of the 2D real transforms of every stage.

def _one_run(case, N, strategy):
    K = (N - 1) // 3
    box = (2 * K + 1) * (K + 1)
    cs = 8 if case["prec"] == "f32" else 16
    nlm, pos = len(_fields(case)) if strategy else 0, 2 if strategy and case.get("pos", True) else 0
    if strategy == 2:
        pos = 2
    eul = nlm if strategy and case.get("eulerian", True) else 0
    base, prod = (3, 2) if _model(case) == "euler2d" else (4, 5)
    trans = base + prod + 3 * (nlm + pos) + (1 if strategy and "q" in _fields(case) else 0)
    st = STAGES[case.get("stepper", "rk4")]
    steps = case["n"]
    state = 2.0 * (3 + nlm + pos + eul) * box * cs * steps
    flops = trans * 2.5 * N * N * 2 * math.log2(N) * st * steps
    outs = (nlm + pos + eul) if strategy else 3
    return state + 8.0 * N * N * (3 + outs), flops


def work(case):
    if case["kind"] == "remap":
        N, nf = int(case["N"]), len(_fields(case))
        # 9 adds and 10 multiplies per component and iteration, 7 per field
        return {"bytes": 8.0 * N * N * (2 + 2 * nf + 3), "flops": 1.0 * N * N * (34 * case["iters"] + 7 * nf)}
    if case["kind"] == "interval":
        runs = [_one_run(case, N, st) for N, st in _runs(case)]
    elif case["kind"] == "steps":
        runs = [_one_run(dict(case, fields=""), int(case["N"]), 0)]
    else:
        N, nf = int(case["N"]), len(_fields(case)) + 2
        b, f = _one_run(dict(case, eulerian=False), N, 0)
        taps = 16 if case["interp"] == "cubic" else 4
        two = 2 if case["scheme"] == "trapezoid" else 1
        # fields and their sources read and written, u, v, h, zeta formed
        runs = [(b + 8.0 * N * N * (case["n"] * (2 * nf + 2 * two * nf + 4) + nf),
                 f + case["n"] * N * N * (2.0 * taps * two * nf + 4 * 2.5 * 2 * math.log2(N)))]
    return {"bytes": float(sum(r[0] for r in runs)), "flops": float(sum(r[1] for r in runs))}


# ---------------------------------------------------------------------------
# The same results in FP64 with plain torch.

class _Exact:
    """Shallow-water (or two-dimensional Euler) run with an averaging
    interval, full-grid real FFTs, all fields stacked in a dict."""

    def __init__(self, case, ic, strategy):
        self.case, self.strategy = case, strategy
        N = self.N = ic.shape[-1]
        self.dt, self.e2 = _dt(N, case), _model(case) == "euler2d"
        self.kx, self.ky = _wavenumbers(N)
        K = (N - 1) // 3
        self.mask = ((self.kx <= K) & (self.ky.abs() <= K)).to(torch.float64)
        self.k2 = self.kx ** 2 + self.ky ** 2
        lap = case.get("visc", "hyper8") == "laplace"
        damp = torch.exp(-_nu(N, case) * (self.k2 if lap else self.k2 ** 4) * self.dt * 0.5)
        one = torch.ones_like(damp)
        y = {"u": self.spec(ic[0]), "v": self.spec(ic[1]), "h": self.spec(ic[2])}
        if not self.e2:
            y["h"][0, 0] -= 1.0
        self.E = {"u": damp, "v": damp, "h": one if lap else damp}
        zero = torch.zeros_like(y["u"])
        self.fields = _fields(case) if strategy else ()
        if strategy:
            names = ["g_" + f for f in self.fields]
            if strategy == 2 or case.get("pos", True):
                names += ["px", "py"]
            for k in names:
                y[k], self.E[k] = zero, damp
            if case.get("eulerian", True) and case["kind"] == "interval":
                for f in self.fields:
                    y["e_" + f], self.E["e_" + f] = zero, one
        self.y = y
        if self.e2:
            self.slave(self.y)

    def spec(self, f):
        return torch.fft.rfft2(f) * (self.mask / (self.N * self.N))

    def phys(self, F):
        return torch.fft.irfft2(F, s=(self.N, self.N)) * float(self.N * self.N)

    def dx(self, F):
        return 1j * self.kx * F

    def dy(self, F):
        return 1j * self.ky * F

    def slave(self, y):
        inv = torch.where(self.k2 > 0, 1.0 / self.k2.clamp_min(1.0), 0.0)
        y["u"], y["v"] = 1j * self.ky * y["h"] * inv, -1j * self.kx * y["h"] * inv

    def sources(self, y):
        """Physical u, v, zeta, eta and the spectra of the averaged scalars."""
        zh = y["h"] if self.e2 else self.dx(y["v"]) - self.dy(y["u"])
        hat = {"zeta": zh, "h": y["h"], "u": y["u"], "v": y["v"]}
        p = {"zeta": self.phys(zh), "h": self.phys(y["h"]), "u": self.phys(y["u"]), "v": self.phys(y["v"])}
        if "q" in self.fields:
            p["q"] = (1.0 + p["zeta"]) / (1.0 + p["h"])
            hat["q"] = self.spec(p["q"])
        return p, hat

    def rhs(self, y, s):
        p, hat = self.sources(y)
        u, v, z, eta = p["u"], p["v"], p["zeta"], p["h"]
        r = {}
        if self.e2:
            r["u"] = r["v"] = torch.zeros_like(y["u"])
            r["h"] = -self.dx(self.spec(u * z)) - self.dy(self.spec(v * z))
        else:
            B = y["h"] + self.spec(0.5 * (u * u + v * v))
            r["u"] = y["v"] + self.spec(z * v) - self.dx(B)
            r["v"] = -y["u"] - self.spec(z * u) - self.dy(B)
            r["h"] = -self.dx(self.spec(u + eta * u)) - self.dy(self.spec(v + eta * v))
        if self.strategy == 1:
            for f in self.fields:
                g = y["g_" + f]
                r["g_" + f] = hat[f] - self.spec(u * self.phys(self.dx(g)) + v * self.phys(self.dy(g)))
            for k, a in (("px", "u"), ("py", "v")):
                if k in y:
                    g = y[k]
                    r[k] = s * hat[a] - self.spec(u * self.phys(self.dx(g)) + v * self.phys(self.dy(g)))
        elif self.strategy == 2:
            xx, xy = self.phys(y["px"]), self.phys(y["py"])
            wx, wy = (xx / s, xy / s) if s > 0 else (0.5 * u, 0.5 * v)
            for k, a, w in (("px", "u", wx), ("py", "v", wy)):
                g = y[k]
                r[k] = self.spec(_interp(p[a], xx, xy, False) - w - wx * self.phys(self.dx(g))
                                 - wy * self.phys(self.dy(g)))
            for f in self.fields:
                g = y["g_" + f]
                r["g_" + f] = self.spec(_interp(p[f], xx, xy, False) - wx * self.phys(self.dx(g))
                                        - wy * self.phys(self.dy(g)))
        for f in self.fields:
            if "e_" + f in y:
                r["e_" + f] = hat[f]
        return r

    def stage(self, y):
        if self.e2:
            self.slave(y)
        return y

    def step(self, n):
        y, E, dt, s = self.y, self.E, self.dt, n * self.dt
        kind = self.case.get("stepper", "rk4")
        a = self.rhs(y, s)
        if kind == "euler":
            self.y = self.stage({k: E[k] ** 2 * (y[k] + dt * a[k]) for k in y})
        elif kind == "heun":
            y1 = self.stage({k: E[k] ** 2 * (y[k] + dt * a[k]) for k in y})
            b = self.rhs(y1, s + dt)
            self.y = self.stage({k: E[k] ** 2 * y[k] + dt / 2 * (E[k] ** 2 * a[k] + b[k]) for k in y})
        else:
            y1 = self.stage({k: E[k] * (y[k] + dt / 2 * a[k]) for k in y})
            b = self.rhs(y1, s + dt / 2)
            y2 = self.stage({k: E[k] * y[k] + dt / 2 * b[k] for k in y})
            c = self.rhs(y2, s + dt / 2)
            y3 = self.stage({k: E[k] ** 2 * y[k] + dt * E[k] * c[k] for k in y})
            d = self.rhs(y3, s + dt)
            self.y = self.stage({k: E[k] ** 2 * y[k] + dt / 6 * (E[k] ** 2 * a[k] + 2 * E[k] * (b[k] + c[k]) + d[k])
                                 for k in y})

    def interval(self):
        n = self.case["n"]
        for i in range(n):
            self.step(i)
        T, X = n * self.dt, _grid(self.N)
        out = {}
        for k in _keys(self.case, self.strategy):
            if k in ("pos_x", "pos_y"):
                d = self.phys(self.y["p" + k[-1]])
                out[k] = X[k == "pos_y"] + (d if self.strategy == 2 else -d / T)
            else:
                f = self.phys(self.y[k if k.startswith("e_") else "g_" + k]) / T
                out[k] = f + 1.0 if k in ("h", "e_h") else f
        return out

    def depth(self):
        u, v, h = (self.phys(self.y[k]) for k in "uvh")
        return torch.stack([u, v, h if self.e2 else h + 1.0])


def _interp(f, dx, dy, cubic):
    """f at grid point + displacement: bilinear or 4-point Lagrange."""
    N = f.shape[-1]
    cx, cy = dx * (N / (2 * math.pi)), dy * (N / (2 * math.pi))
    fx, fy = torch.floor(cx), torch.floor(cy)
    ax, ay = cx - fx, cy - fy
    n = torch.arange(N, device=f.device)
    i0, j0 = n[None, :] + fx.long(), n[:, None] + fy.long()
    if cubic:
        def w(a):
            return (-a * (a - 1) * (a - 2) / 6, (a + 1) * (a - 1) * (a - 2) / 2, -(a + 1) * a * (a - 2) / 2,
                    (a + 1) * a * (a - 1) / 6)
        wx, wy, lo = w(ax), w(ay), -1
    else:
        wx, wy, lo = (1 - ax, ax), (1 - ay, ay), 0
    out = torch.zeros_like(dx)
    for b, wb in enumerate(wy):
        row = ((j0 + b + lo) % N) * N
        for a, wa in enumerate(wx):
            out += wa * wb * f.reshape(-1)[row + (i0 + a + lo) % N]
    return out


def _exact_sl(case, ic):
    m = _Exact(dict(case, kind="steps"), ic, 0)
    m.fields = _fields(case)  # q among the sources
    dt, n, trap, cubic = m.dt, case["n"], case["scheme"] == "trapezoid", case["interp"] == "cubic"

    def physical():
        p, _ = m.sources(m.y)
        return dict(p, h=p["h"] + 1.0)

    g = {f: torch.zeros_like(ic[0]) for f in m.fields}
    d = [torch.zeros_like(ic[0]), torch.zeros_like(ic[0])]
    old = physical()
    for i in range(n):
        m.step(i)
        p = physical()
        at = (-dt * p["u"], -dt * p["v"], cubic)
        for f in m.fields:
            src = 0.5 * (_interp(old[f], *at) + p[f]) if trap else p[f]
            g[f] = _interp(g[f], *at) + dt * src
        c = (i * dt + (0.5 * dt if trap else 0.0)) * dt
        d = [_interp(d[0], *at) + c * p["u"], _interp(d[1], *at) + c * p["v"]]
        old = p
    X, Y = _grid(m.N)
    T = n * dt
    return dict({f: g[f] / T for f in m.fields}, pos_x=X - d[0] / T, pos_y=Y - d[1] / T)


def _exact_remap(case, seed):
    pos, src = _remap_inputs(case, seed)
    X, Y = _grid(int(case["N"]))
    dx, dy = X - pos[0], Y - pos[1]
    xx = xy = torch.zeros_like(dx)
    for _ in range(case["iters"]):
        nx, ny = _interp(dx, xx, xy, False), _interp(dy, xx, xy, False)
        resid = torch.maximum((nx - xx).abs(), (ny - xy).abs())
        xx, xy = nx, ny
    out = {k: _interp(f, xx, xy, False) for k, f in src.items()}
    # the residual of a converged iteration is rounding: no value of its own
    return dict(out, xi_x=X + xx, xi_y=Y + xy, resid=resid if float(resid.max()) > 1e-6 else None)


def exact(case, seed):
    if case["kind"] == "remap":
        return _exact_remap(case, seed)
    ics = _initials(case, seed)
    if case["kind"] == "sl":
        return [_exact_sl(case, ics[0])]
    if case["kind"] == "steps":
        m = _Exact(case, ics[0], 0)
        for i in range(case["n"]):
            m.step(i)
        return m.depth()
    out = [_Exact(case, ic, st).interval() for ic, (_, st) in zip(ics, _runs(case))]
    return out if len(out) <= 4 else [torch.stack(list(o.values())) for o in out]
