"""The workloads this library is timed on: whole calls of its public entry points (the Solver, the
batched sweep, the allocation-free step) over the sizes, precisions, limiters, media and boundaries
that its users run.

`listed()` names them, `draw(rng)` gives further ones of the same ranges, `prepare` makes what a
caller holds before the call, `run` is one call, `work` its unavoidable traffic and arithmetic and
`exact` its result in plain 64-bit torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1805_03442_gb300 import inputs, sv

PREC = {"fp32": sv.FP32, "fp64": sv.FP64, "fp32_p64": sv.FP32_P64, "fp32_pc": sv.FP32_PC,
        "fp32_ps": sv.FP32_PS}
LIM = {"minmod": sv.MINMOD, "vanleer": sv.VANLEER, "mc": sv.MC}
GAMMA = 1.4
# arithmetic of one cell's step (slopes, predictor, one HLL face per axis, source twice, bound)
FLOPS = {1: 300, 2: 560, 3: 900}


def listed():
    return [
        # the smallest call: one step between the caller's own device buffers, dt read back
        # (a host code that owns its memory and steps the library itself)
        {"name": "noalloc_1000_fp32", "kind": "noalloc", "n": 1000, "prec": "fp32", "lim": "minmod"},
        # the paper's one-wavelength linear stage at 1024 cells: upload, run to a time, download
        {"name": "wave_1024_fp32", "kind": "wave", "n": 1024, "prec": "fp32", "lim": "minmod",
         "t_end": 0.25},
        # the same study in double on the paper's largest 1D grid (N = 200 ... 1600), where the
        # growth of an eigenmode is followed far below float's noise
        {"name": "wave_1600_fp64", "kind": "wave", "n": 1600, "prec": "fp64", "lim": "vanleer",
         "t_end": 0.1},
        # the paper's colliding shocks between walls on its 10^5-cell reference grid (frozen gas)
        {"name": "shocks_100000_fp32", "kind": "shocks", "n": 100000, "prec": "fp32",
         "lim": "minmod", "steps": 512},
        # the paper's forced source: a wave driven at x = 0 into the active gas, free outflow, in
        # the perturbation layout that such small signals ask for
        {"name": "forced_65536_ps", "kind": "forced", "n": 65536, "prec": "fp32_ps",
         "lim": "minmod", "steps": 256},
        # the benchmark's broad spectrum, 2^22 cells: upload, 64 steps, download
        {"name": "spectrum_4194304_fp32", "kind": "spectrum", "n": 1 << 22, "prec": "fp32",
         "lim": "minmod", "steps": 64},
        # a large 1D run in double, the accuracy reference of every float run
        {"name": "spectrum_1000000_fp64", "kind": "spectrum", "n": 1000000, "prec": "fp64",
         "lim": "minmod", "steps": 8},
        # the 2D benchmark grid: an oblique plane wave with noise, state left on the device
        {"name": "plane_8192x8192_fp32", "kind": "plane", "nx": 8192, "ny": 8192, "prec": "fp32",
         "lim": "minmod", "steps": 32},
        # the paper's 2D active sector (medium map, pulsating source, wall and outflow), in double
        {"name": "sector_500_fp64", "kind": "sector", "nx": 500, "prec": "fp64", "lim": "minmod",
         "steps": 16},
        # the 3D benchmark grid: a random field, state left on the device
        {"name": "random_512_fp32", "kind": "random3d", "nx": 512, "ny": 512, "nz": 512,
         "prec": "fp32", "lim": "minmod", "steps": 8},
        # 3D with the double-accuracy pressure recovery, on a box of unequal odd sides
        {"name": "random_201x150x170_p64", "kind": "random3d", "nx": 201, "ny": 150, "nz": 170,
         "prec": "fp32_p64", "lim": "minmod", "steps": 8},
        # a stability map: 256 runs of uneven sizes and media, from upload to the states and mode
        # logs of every run
        {"name": "sweep_256_fp32", "kind": "sweep", "runs": 256, "n_lo": 256, "n_hi": 6000,
         "prec": "fp32", "lim": "minmod", "draw": 2026},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["noalloc", "wave", "shocks", "forced", "spectrum", "plane", "sector",
                       "random3d", "sweep"])
    lim = rng.choice(["minmod", "minmod", "vanleer", "mc"])
    prec = rng.choice(["fp32", "fp32", "fp64", "fp32_p64", "fp32_pc", "fp32_ps"])
    slow = prec in ("fp64", "fp32_p64")
    if kind == "noalloc":
        return {"kind": kind, "n": _log(rng, 100, 300000), "lim": lim,
                "prec": rng.choice(["fp32", "fp64", "fp32_p64", "fp32_pc"])}
    if kind == "wave":
        n = _log(rng, 200, 16000)
        return {"kind": kind, "n": n, "prec": prec, "lim": "vanleer" if prec == "fp64" else lim,
                "t_end": min(0.25, 300.0 / n)}
    if kind in ("shocks", "forced"):
        if kind == "shocks" and prec == "fp32_ps":
            prec = "fp32"           # the layout of small perturbations is not for strong shocks
        n = _log(rng, 1000, 200000)
        return {"kind": kind, "n": n, "prec": prec, "lim": "minmod",
                "steps": rng.randint(32, 64) if slow else rng.randint(100, 600)}
    if kind == "spectrum":
        n = _log(rng, 1 << 17, (1 << 20) if slow else (1 << 22))
        return {"kind": kind, "n": n, "prec": prec, "lim": lim, "steps": rng.randint(8, 64) // (4 if slow else 1)}
    if kind == "plane":
        top = 2000 if slow else 6000
        return {"kind": kind, "nx": _log(rng, 64, top), "ny": _log(rng, 64, top), "prec": prec,
                "lim": lim, "steps": rng.randint(8, 24) // (4 if slow else 1)}
    if kind == "sector":
        return {"kind": kind, "nx": _log(rng, 100, 600 if slow else 2048), "prec": prec,
                "lim": "minmod", "steps": rng.randint(16, 64) // (4 if slow else 1)}
    if kind == "random3d":
        top = 150 if slow else 320
        return {"kind": kind, "nx": _log(rng, 20, top), "ny": _log(rng, 20, top),
                "nz": _log(rng, 20, top), "prec": prec, "lim": lim,
                "steps": rng.randint(4, 12) // (2 if slow else 1)}
    lo = rng.randint(100, 1000)
    return {"kind": "sweep", "runs": _log(rng, 16, 400), "n_lo": lo, "n_hi": lo + rng.randint(100, 4000),
            "prec": rng.choice(["fp32", "fp32", "fp32_pc", "fp32_ps"]), "lim": lim,
            "draw": rng.randint(1, 10 ** 6)}


# ------------------------------------------------------------------ the problems

def _dims(case):
    k = case["kind"]
    if k == "sector":
        return (case["nx"], case["nx"])
    if k == "plane":
        return (case["nx"], case["ny"])
    if k == "random3d":
        return (case["nx"], case["ny"], case["nz"])
    return (case["n"],)


def _params(case):
    """The media of the repository's own runs of each kind."""
    k, over = case["kind"], {}
    if k in ("wave", "spectrum", "noalloc"):
        over = dict(S=1.0, tau0=0.08)
    elif k == "shocks":
        over = dict(S=0.0, tau0=math.inf)
    elif k == "forced":
        over = dict(S=0.5, tau0=0.0135)
    elif k == "plane":
        over = dict(S=1.0, tau0=0.01)
    elif k == "sector":
        over = dict(S=1.0, tau0=0.0135)
    elif k == "random3d":
        over = dict(S=1.0, tau0=0.08, cfl=0.3)
    return sv.Params(precision=PREC[case["prec"]], limiter=LIM[case["lim"]], **over)


def _length(case):
    if case["kind"] == "sector":
        return 0.2 + math.sqrt(GAMMA)
    return case["n"] / 1024.0 if case["kind"] == "spectrum" else 1.0


def _bc(case):
    return {"shocks": (1, 1), "forced": (3, 2), "sector": (2, 1, 2, 2)}.get(case["kind"], (0, 0))


def _pack(rho, vel, p, ev):
    """Primitive fields (device, float64) -> conserved (nf, ...) state, eq. 5."""
    kin = sum(v * v for v in vel)
    Ev = rho * ev
    return torch.stack([rho] + [rho * v for v in vel] + [p / (GAMMA - 1.0) + 0.5 * rho * kin + Ev, Ev])


def _initial(case, seed):
    """The initial state, float64 (nf, ncell) on the device."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    k, n, P, L = case["kind"], _dims(case), _params(case), _length(case)
    dev, f8 = "cuda", torch.float64
    ev0, c = P.Ck + P.S, math.sqrt(GAMMA)

    def rand(*shape):
        return torch.rand(*shape, generator=g, device=dev, dtype=f8)

    if k in ("wave", "spectrum", "noalloc"):
        # acoustic waves with random phases and a k^-1 spectrum on the uniform equilibrium
        N = n[0]
        modes, m0, amp = (64, max(1, N // 32768), 1e-3) if k == "spectrum" else (4, 1, 1e-3)
        x = (torch.arange(N, device=dev, dtype=f8) + 0.5) / N
        w = torch.zeros(N, device=dev, dtype=f8)
        ph = (2 * math.pi * rand(modes)).tolist()
        for i in range(modes):
            m = m0 * (1 + i)
            w += amp / (1 + i) * torch.cos(2 * math.pi * m * x + ph[i])
        return _pack(1 + w, [c * w], 1 + c * c * w, torch.full_like(w, ev0))
    if k == "shocks":
        N = n[0]
        x = (torch.arange(N, device=dev, dtype=f8) + 0.5) / N
        a, b = [float(v) for v in (0.08 + 0.04 * rand(1))] + [float(v) for v in (0.88 + 0.04 * rand(1))]
        p = torch.where(x < a, 1000.0, torch.where(x < b, 0.01, 100.0)).to(f8)
        one = torch.ones_like(x)
        return _pack(one, [0 * x], p, ev0 * one)
    if k == "forced":
        w = 1e-4 * (rand(n[0]) - 0.5)      # weak noise in the gas at rest
        return _pack(1 + w, [0 * w], 1 + w, torch.full_like(w, ev0))
    if k == "plane":
        nx, ny = n
        h = L / nx
        X = ((torch.arange(nx, device=dev, dtype=f8) + 0.5) * h)[None, :]
        Y = ((torch.arange(ny, device=dev, dtype=f8) + 0.5) * h)[:, None]
        kx, ky = 2 * math.pi * 7 / L, 2 * math.pi * 4 / (ny * h)
        kk = math.hypot(kx, ky)
        w = 1e-3 * torch.cos(kx * X + ky * Y + 2 * math.pi * float(rand(1)))
        rho = 1 + w + 1e-5 * torch.randn(ny, nx, generator=g, device=dev, dtype=f8)
        p = 1 + c * c * w + 1e-5 * torch.randn(ny, nx, generator=g, device=dev, dtype=f8)
        return _pack(rho, [c * w * kx / kk, c * w * ky / kk], p, torch.full_like(w, ev0)).reshape(5, -1)
    if k == "sector":
        nx, ny = n
        w = 1e-4 * (rand(ny, nx) - 0.5)
        return _pack(1 + w, [0 * w, 0 * w], 1 + w, torch.full_like(w, ev0)).reshape(5, -1)
    # 3D: isotropic random density and velocity of rms 1e-3 with a k^-2 power spectrum
    nx, ny, nz = n
    f4 = torch.float32
    kz = torch.fft.fftfreq(nz, 1.0 / nz, device=dev, dtype=f4)[:, None, None]
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device=dev, dtype=f4)[None, :, None]
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, device=dev, dtype=f4)[None, None, :]
    ak = (kx * kx + ky * ky + kz * kz).clamp_min(1.0).rsqrt()

    def field():
        z = torch.fft.irfftn(torch.fft.rfftn(torch.randn(nz, ny, nx, generator=g, device=dev, dtype=f4)) * ak,
                             s=(nz, ny, nx)).reshape(-1)
        return (z * (1e-3 / z.square().mean().sqrt())).to(f8)
    r = field()
    return _pack(1 + r, [c * field() for _ in range(3)], 1 + c * c * r, torch.full_like(r, ev0))


def _drive(case):
    """The wave of the forced run: wavelength 0.1, frozen acoustic, 1e-3."""
    P, c = _params(case), math.sqrt(GAMMA)
    ev0, k = P.Ck + P.S, 2 * math.pi / 0.1
    base = [1.0, 0.0, 1.0 / (GAMMA - 1.0) + ev0, ev0]
    amp = [1e-3, 1e-3 * c, 1e-3 * (c * c / (GAMMA - 1.0) + ev0), 1e-3 * ev0]
    return k * c, complex(k, -3.0), base, amp


class _Run:
    pass


def _sweep_runs(case):
    """Media and sizes of a stability map (seeded by the case: they set its work)."""
    rng = np.random.default_rng(case["draw"])
    out = []
    for _ in range(case["runs"]):
        r = _Run()
        r.n, r.m = int(rng.integers(case["n_lo"], case["n_hi"] + 1)), int(rng.integers(1, 9))
        r.tau0, r.S = float(10.0 ** rng.uniform(-1.5, 1.0)), float(rng.uniform(0.0, 1.0))
        r.tau_rho, r.tau_T = float(rng.uniform(-2.0, 0.0)), float(rng.uniform(-2.5, 0.0))
        r.Q_rho, r.Q_T, r.I_rho, r.I_T = (float(v) for v in rng.uniform(-1.0, 1.0, 4))
        r.L, r.t_end = 1.0, 0.25 / (r.m * math.sqrt(GAMMA))
        out.append(r)
    return out


def _sweep_states(case, seed, runs):
    rng = np.random.default_rng(seed)
    P, out = _params(case), []
    for r in runs:
        md = inputs.Mode(m=r.m, shape=inputs.acoustic_shape(GAMMA),
                         scale=1e-3 * np.exp(2j * math.pi * rng.random()))
        out.append(inputs.waves_1d(GAMMA, r.n, 1.0, (1.0, 1.0, P.Ck + r.S), [md]))
    return out


def _is64(case):
    return case["prec"] == "fp64"


class _View:
    """The solver's own device state as an array (sv_state_device); keeps the solver alive."""

    def __init__(self, solver, ptr, shape, f64):
        self.solver = solver
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f8" if f64 else "<f4",
                                         "data": (ptr, False), "strides": None, "version": 3}


def prepare(case, seed):
    st = {"case": case}
    P = _params(case)
    if case["kind"] == "sweep":
        runs = _sweep_runs(case)
        st["states"] = _sweep_states(case, seed, runs)
        st["batch"] = sv.Batch(P, runs, st["states"], log_cap=32)
        st["n"] = [r.n for r in runs]
        return st
    U = _initial(case, seed)
    host = torch.float64 if _is64(case) or case["prec"] == "fp32_ps" else torch.float32
    if case["kind"] == "noalloc":
        st["P"] = P
        st["in"] = U.to(torch.float64 if _is64(case) else torch.float32).contiguous()
        st["out"] = torch.empty_like(st["in"])
        return st
    # a caller that stages through page-locked memory
    st["in"] = torch.empty(U.shape, dtype=host, pin_memory=True)
    st["in"].copy_(U)
    if len(_dims(case)) == 1:
        st["out"] = torch.empty(U.shape, dtype=host, pin_memory=True)
    n, L = _dims(case), _length(case)
    s = sv.Solver(P, n, tuple(L * m / n[0] for m in n), bc=_bc(case))
    if case["kind"] == "forced":
        s.set_drive(*_drive(case))
    if case["kind"] == "sector":
        q = inputs.sector_problem(case["nx"])
        s.set_medium2d(*q.maps, omega=q.omega, amp=q.amp)
    st["solver"] = s
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    t32 = (lambda t: t) if _is64(case) else (lambda t: torch.tensor(t, dtype=torch.float32))
    if kind == "sweep":
        b = st["batch"]
        b.reset(st["states"])
        b.run()
        b.sync()
        U, t, k, fl, log = [], [], [], [], []
        for i in range(len(st["n"])):
            u, ti, ki, fi = b.read(i)
            tl, am = b.mode_log(i)
            U.append(u.reshape(-1))
            t.append(ti)
            k.append(ki)
            fl.append(fi)
            log += [am.real, am.imag]
        return {"state": np.concatenate(U).astype(np.float32), "t": np.array(t, dtype=np.float32),
                "steps": np.array(k), "flags": np.array(fl, dtype=np.int64),
                "log": np.concatenate(log).astype(np.float32)}
    if kind == "noalloc":
        dt, flags = sv.step1d_noalloc(st["P"], case["n"], 1.0, st["in"].data_ptr(), st["out"].data_ptr())
        return {"state": st["out"], "dt": t32(dt), "flags": flags}
    s = st["solver"]
    wide = st["in"].dtype == torch.float64
    (s.write_state_ptr if wide else s.write_state_ptr_f32)(st["in"].data_ptr())
    steps = None
    if "t_end" in case:
        _, steps = s.run_to(case["t_end"])
    else:
        s.step(case["steps"])
    if s.dim == 1 and case["prec"] != "fp32_ps":
        t = (s.read_state_ptr if wide else s.read_state_ptr_f32)(st["out"].data_ptr())
        out = st["out"]
    else:
        ptr, _ = s.state_device()
        out = torch.as_tensor(_View(s, ptr, (s.nf, s.ncell), _is64(case)), device="cuda")
        t = s.time()[0]
    got = {"state": out, "t": t32(t), "flags": s.status()}
    if steps is not None:
        got["steps"] = steps
    return got


def work(case):
    kind = case["kind"]
    if kind == "sweep":
        b = f = 0.0
        for r in _sweep_runs(case):
            steps = r.t_end / (0.4 / r.n / math.sqrt(GAMMA))
            b += 2 * 16 * r.n
            f += FLOPS[1] * r.n * steps
        return {"bytes": b, "flops": f}
    n = _dims(case)
    cells = math.prod(n)
    steps = case.get("steps", 1)
    if "t_end" in case:
        steps = case["t_end"] / (0.4 * _length(case) / n[0] / math.sqrt(GAMMA))
    state = cells * (len(n) + 3) * (8 if _is64(case) else 4)
    # every step's dt depends on the whole state before it: a state larger than the on-chip
    # memories passes through HBM once each way per step; a smaller one is read and written once
    passes = steps if 2 * state > 126e6 else 1
    return {"bytes": 2.0 * state * passes, "flops": float(FLOPS[len(n)]) * cells * steps}


# ------------------------------------------------------------------ 64-bit results

def _limit(lim, a, b):
    same = a * b > 0
    if lim == "minmod":
        m = torch.minimum(a.abs(), b.abs())
    elif lim == "vanleer":
        m = 2 * a * b / (a + b).abs().clamp_min(1e-300)
    else:
        m = torch.minimum(2 * torch.minimum(a.abs(), b.abs()), 0.5 * (a + b).abs())
    return torch.where(same, torch.copysign(m, a), torch.zeros_like(a))


class _Gas:
    """The scheme's formulas (eqs. 5-7, 13-16) in float64; parameters numbers or per-cell tensors."""

    def __init__(self, P, dim, frozen, per=None):
        self.dim, self.P, self.frozen = dim, P, frozen
        q = per or P
        self.S, self.tau0 = q.S, q.tau0
        self.ex = (q.tau_rho, q.tau_T, q.Q_rho, q.Q_T, q.I_rho, q.I_T)
        self.plain = per is None and not any(self.ex[2:])

    def prim(self, u):
        d = self.dim
        v = [u[1 + a] / u[0] for a in range(d)]
        kin = sum(u[1 + a] * v[a] for a in range(d))
        return v, (GAMMA - 1.0) * (u[1 + d] - 0.5 * kin - u[2 + d])

    def power(self, rho, T, a, b):
        return torch.exp(a * torch.log(rho) + b * torch.log(T))

    def source(self, u):
        if self.frozen:
            return None
        d = self.dim
        _, p = self.prim(u)
        rho, T = u[0], p / u[0]
        itau = self.power(rho, T, -self.ex[0], -self.ex[1]) / self.tau0
        Q0 = self.S / self.tau0
        Q = I = Q0
        if not self.plain:
            Q = Q0 * self.power(rho, T, self.ex[2], self.ex[3])
            I = Q0 * self.power(rho, T, self.ex[4], self.ex[5])
        return (0.0 if self.plain else rho * (Q - I)), (self.P.Ck * p - u[2 + d]) * itau + rho * Q

    def flux(self, u, v, p, a):
        d = self.dim
        return torch.stack([u[1 + a]] + [u[1 + b] * v[a] + (p if b == a else 0.0) for b in range(d)] +
                           [v[a] * (u[1 + d] + p), v[a] * u[2 + d]])

    def hll(self, L, R, cl, cr, a):
        vl, pl = self.prim(L)
        vr, pr = self.prim(R)
        bad = ~((L[0] > 0) & (pl > 0) & (R[0] > 0) & (pr > 0))
        if bool(bad.any()):
            L, R = torch.where(bad, cl, L), torch.where(bad, cr, R)
            vl, pl = self.prim(L)
            vr, pr = self.prim(R)
        a_l, a_r = torch.sqrt(GAMMA * pl / L[0]), torch.sqrt(GAMMA * pr / R[0])
        sl = torch.minimum(vl[a] - a_l, vr[a] - a_r).clamp_max(0.0)
        sr = torch.maximum(vl[a] + a_l, vr[a] + a_r).clamp_min(0.0)
        return (sr * self.flux(L, vl, pl, a) - sl * self.flux(R, vr, pr, a) + sl * sr * (R - L)) / (sr - sl)

    def bounds(self, u):
        """Per cell: signal speed of eq. 16 and tau (None in the frozen gas)."""
        v, p = self.prim(u)
        vm = v[0].abs() if self.dim == 1 else torch.sqrt(sum(x * x for x in v))
        s = torch.maximum(2 * vm, vm + torch.sqrt(GAMMA * p / u[0]))
        tau = None if self.frozen else self.tau0 * self.power(u[0], p / u[0], self.ex[0], self.ex[1])
        return s, tau

    def step(self, U, shift, dt, h, lim, active=None):
        """One step of a padded state: shift(x, a, k) moves by k cells along axis a."""
        d = self.dim
        div, slopes, ok = 0.0, [], None
        for a in range(d):
            s = _limit(lim, U - shift(U, a, -1), shift(U, a, 1) - U)
            A, B = U + 0.5 * s, U - 0.5 * s
            va, pa = self.prim(A)
            vb, pb = self.prim(B)
            good = (A[0] > 0) & (pa > 0) & (B[0] > 0) & (pb > 0)
            ok = good if ok is None else ok & good
            div = div + self.flux(A, va, pa, a) - self.flux(B, vb, pb, a)
            slopes.append(s)
            del A, B, va, vb, pa, pb
        zero = torch.zeros((), dtype=U.dtype, device=U.device)
        div = torch.where(ok, div, zero)
        slopes = [torch.where(ok, s, zero) for s in slopes]
        W = U - (0.5 * dt / h) * div

        def add(X, Y, f):
            if Y is None:
                return X
            for i, y in ((1 + d, Y[0]), (2 + d, Y[1])):
                if torch.is_tensor(y):
                    X[i] += f * (y if active is None else torch.where(active, y, zero))
            return X
        W = add(W, self.source(U), 0.5 * dt)
        N = U.clone()
        for a in range(d):
            F = self.hll(shift(W + 0.5 * slopes[a], a, -1), W - 0.5 * slopes[a], shift(U, a, -1), U, a)
            N -= (dt / h) * (shift(F, a, 1) - F)
            del F
        return add(N, self.source(W), dt)


def _exact_grid(case, seed):
    """A solver's run on its grid, by whole-array 64-bit torch operations."""
    P, n, L, kind = _params(case), _dims(case), _length(case), case["kind"]
    d, h = len(n), L / n[0]
    gas = _Gas(P, d, math.isinf(P.tau0))
    U = _initial(case, seed)
    if not _is64(case):
        U = U if case["prec"] == "fp32_ps" else U.float().double()
    U = U.reshape((d + 3,) + tuple(reversed(n)))
    bc = _bc(case)
    walled = any(bc)
    active = driven = None
    if kind == "sector":
        q = inputs.sector_problem(case["nx"])
        col = torch.arange(n[0], device=U.device)[None, :]
        lo, hi, dlo, dhi = (torch.from_numpy(m).to(U.device)[:, None] for m in q.maps)
        active, driven = (col >= lo) & (col < hi), (col >= dlo) & (col < dhi)

    def shift(x, a, k):
        return torch.roll(x, -k, dims=x.dim() - 1 - a)

    def ghosts(x, t):
        """Two ghost cells per side of every axis that is not periodic."""
        for a in range(d):
            ax = x.dim() - 1 - a

            def side(which, b):
                m = x.shape[ax]
                if b == 1:
                    idx = [1, 0] if which == 0 else [m - 1, m - 2]
                elif b == 2:
                    idx = [0, 0] if which == 0 else [m - 1, m - 1]
                else:
                    idx = [m - 2, m - 1] if which == 0 else [0, 1]
                g = x.index_select(ax, torch.tensor(idx, device=x.device))
                if b == 1 and x.dtype != torch.bool:
                    g[1 + a] = -g[1 + a]
                if b == 3:
                    om, kc, base, amp = _drive(case)
                    for i, j in enumerate((-2, -1)):
                        ph = np.exp(1j * (kc * (j + 0.5) * h - om * t))
                        for f in range(4):
                            g[f, i] = base[f] + (amp[f] * ph).real
                return g
            x = torch.cat([side(0, bc[2 * a]), x, side(1, bc[2 * a + 1])], dim=ax)
        return x

    act = None
    if active is not None:
        act = ghosts(active[None], 0.0)[0]
    t, k, t_end = 0.0, 0, case.get("t_end", math.inf)
    while t < t_end and k < case.get("steps", 1 if kind == "noalloc" else 1 << 60):
        s, tau = gas.bounds(U)
        dt = P.cfl * h / float(s.max())
        if tau is not None:
            dt = min(dt, P.c_tau * float(tau.min()))
        del s, tau
        last = dt >= t_end - t
        if last:
            dt = t_end - t
        if walled:
            X = gas.step(ghosts(U, t), shift, dt, h, case["lim"], act)
            U = X[(slice(None),) + (slice(2, -2),) * d].contiguous()
        elif d > 1 and U.numel() > 1 << 26:
            # slabs along the last axis (with the two planes either side that a step reads)
            # bound the memory
            out, m = torch.empty_like(U), max(1, (1 << 24) // math.prod(n[:-1]))
            for z in range(0, n[-1], m):
                idx = torch.arange(z - 2, min(z + m, n[-1]) + 2, device=U.device) % n[-1]
                out[:, z:z + m] = gas.step(U[:, idx], shift, dt, h, case["lim"])[:, 2:-2]
            U = out
        else:
            U = gas.step(U, shift, dt, h, case["lim"])
        t = t_end if last else t + dt
        k += 1
        if driven is not None:
            w = q.amp * math.sin(q.omega * t)
            cell = [1 + w, 0.0, 0.0, (1 + GAMMA * w) / (GAMMA - 1.0) + (1 + w) * (P.Ck + P.S), (1 + w) * (P.Ck + P.S)]
            for f in range(5):
                U[f] = torch.where(driven, torch.tensor(cell[f], dtype=U.dtype, device=U.device), U[f])
    U = U.reshape(d + 3, -1)
    if case["prec"] == "fp32_ps":
        ev0 = P.Ck + P.S
        U[0] -= 1.0
        U[1 + d] -= 1.0 / (GAMMA - 1.0) + ev0
        U[2 + d] -= ev0
    return {"state": U, "dt" if kind == "noalloc" else "t": t}


def _exact_sweep(case, seed):
    """All runs at once: their cells in one row, neighbours by index, one dt per run."""
    runs = _sweep_runs(case)
    P, dev = _params(case), "cuda"
    states = _sweep_states(case, seed, runs)
    U = torch.from_numpy(np.concatenate(states, axis=1)).to(dev)
    if case["prec"] != "fp32_ps":
        U = U.float().double()
    n = np.array([r.n for r in runs])
    off = np.concatenate([[0], np.cumsum(n)[:-1]])
    rid = torch.from_numpy(np.repeat(np.arange(len(n)), n)).to(dev)
    here = torch.arange(int(n.sum()), device=dev)
    first, size = torch.from_numpy(off).to(dev)[rid], torch.from_numpy(n).to(dev)[rid]
    index = {-1: first + (here - first - 1) % size, 1: first + (here - first + 1) % size}

    def shift(x, a, k):
        return x[..., index[k]]

    per = _Run()
    for f in ("S", "tau0", "tau_rho", "tau_T", "Q_rho", "Q_T", "I_rho", "I_T"):
        setattr(per, f, torch.tensor([getattr(r, f) for r in runs], dtype=torch.float64, device=dev)[rid])
    gas = _Gas(P, 1, False, per)
    h = torch.tensor([1.0 / r.n for r in runs], dtype=torch.float64, device=dev)
    t_end = torch.tensor([r.t_end for r in runs], dtype=torch.float64, device=dev)
    t = torch.zeros_like(t_end)
    zero = torch.zeros_like(t_end)
    while bool((t < t_end).any()):
        s, tau = gas.bounds(U)
        smax = zero.scatter_reduce(0, rid, s, "amax")
        tmin = torch.full_like(zero, math.inf).scatter_reduce(0, rid, tau, "amin")
        dt = torch.minimum(P.cfl * h / smax, P.c_tau * tmin)
        rest = t_end - t
        last = dt >= rest
        dt = torch.where(last, rest, dt)
        U = torch.where((dt > 0)[rid], gas.step(U, shift, dt[rid], h[rid], case["lim"]), U)
        t = torch.where(last, t_end, t + dt)
    parts = torch.split(U, n.tolist(), dim=1)
    return {"state": torch.cat([p.reshape(-1) for p in parts]), "t": t, "steps": None, "flags": None, "log": None}


def exact(case, seed):
    return _exact_sweep(case, seed) if case["kind"] == "sweep" else _exact_grid(case, seed)
