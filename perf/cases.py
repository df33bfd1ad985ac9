"""The performance cases of this repository: what a user has the framework do, through its
public entry points (``lbkm.Solver``, ``lbkm.Solver.batched``, ``lbkm.Solver24``).

A pass starts a run from fields that the user holds on the GPU (``init_fields``), advances it
(``step``) and takes the result: the macroscopic fields of an FP64 run (``macros``), the state
planes of an FP32 run (``planes_device``), and the TNE records where the run keeps them
(``tne_history``). The gradient cases call ``grad`` in place of ``step``.

``exact`` is an independent FP64 statement of the model (arXiv:1411.6697) in whole-array torch
operations: dense moment matrices, flux differences with minmod, and reverse-mode
differentiation for the gradient.
"""
import math

import numpy as np
import torch

from paper_1411_6697_gb300 import lbkm

DEV = "cuda"
F8 = torch.float64
L2_BYTES = 126e6      # a state that fits on the chip need not leave it between steps
GAMMA = 1.4           # I = 3, the value of the paper's detonations
SETS24 = ((2.7, 2.2, 1.2), (5.0, 3.0, 1.1))    # D2V24 of the steady detonation
ORBITS16 = ((2.7, 5.0), (2.2, 0.0), (1.2, 3.0), (1.0, 0.0))
# the regular shock reflection's velocity set and side states (rho, ux, uy, T)
ORBITS16_REFLECTION = ((3.0, 2.5), (2.9, 0.0), (1.0, 1.5), (1.0, 0.0))
INFLOW, LID = (1.0, 2.0, 0.0, 0.5), (1.25, 1.9, -0.173205, 0.56)


def listed():
    return [
        # the Sod tube at the size and length the paper runs it: the smallest grid, where the
        # latency of one step after another is everything
        dict(name="sod_400_f64", kind="sod", nx=400, ny=1, steps=1000, f64=True, tne=0),
        # the steady-detonation run with its TNE records taken at every step, plain FP64
        dict(name="detonation_16384_f64_tne", kind="detonation", nx=16384, ny=1, steps=128,
             f64=True, tne=1),
        # the same run in FP32 without records: a long march to the steady state
        dict(name="detonation_16384_f32", kind="detonation", nx=16384, ny=1, steps=512,
             f64=False, tne=0),
        # the 2-D reactive field with TNE records, FP32: the headline workload, largest grid
        dict(name="field_4096_f32_tne", kind="field", nx=4096, ny=4096, steps=32, f64=False,
             tne=1, df32=False, equal=False),
        # a ragged, odd-sized field without records, double-float recovery
        dict(name="field_1030x517_f32", kind="field", nx=1030, ny=517, steps=96, f64=False,
             tne=0, df32=True, equal=False),
        # the single-relaxation-time comparison run: all rates equal, FP32
        dict(name="field_2048_f32_equal", kind="field", nx=2048, ny=2048, steps=32, f64=False,
             tne=0, df32=False, equal=True),
        # the FP64 field a user checks the FP32 one against
        dict(name="field_1024_f64", kind="field", nx=1024, ny=1024, steps=8, f64=True, tne=0,
             df32=False, equal=False),
        # regular shock reflection (fixed inflow and lid, outflow, reflecting floor)
        dict(name="reflection_300x100_f32", kind="reflection", nx=300, ny=100, steps=64,
             f64=False, tne=0),
        # a parameter study: 512 detonations of uneven length, own rates and heat release
        dict(name="batched_512_f32", kind="batched", n=512, nx_min=1024, nx_max=65536, steps=64),
        # sensitivities of a detonation: one gradient call with checkpoints every 64 steps
        dict(name="gradient_8192x256", kind="gradient", nx=8192, steps=256),
        # the paper's own 24-velocity model: its steady detonation in FP64, and a 2-D field
        dict(name="d2v24_detonation_5000_f64", kind="detonation24", nx=5000, ny=1, steps=256,
             f64=True, tne=0),
        dict(name="d2v24_field_2048_f32", kind="field24", nx=2048, ny=2048, steps=6, f64=False,
             tne=0, df32=False, equal=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds: sizes over the whole range, odd ones among them."""
    kind = rng.choice(["sod", "detonation", "detonation", "field", "field", "field", "reflection",
                       "batched", "gradient", "detonation24", "field24", "field24"])
    if kind == "batched":
        hi = _log(rng, 2048, 65536)
        return dict(kind=kind, n=_log(rng, 8, 480), nx_min=max(64, hi // rng.choice([1, 8, 64])),
                    nx_max=hi, steps=rng.randint(20, 60))
    if kind == "gradient":
        return dict(kind=kind, nx=_log(rng, 256, 8192), steps=rng.randint(65, 250))
    f64 = rng.random() < 0.4
    tne = 1 if rng.random() < 0.35 else 0
    if kind == "sod":
        return dict(kind=kind, nx=_log(rng, 100, 4000), ny=1, steps=rng.randint(64, 900), f64=f64,
                    tne=0)
    if kind in ("detonation", "detonation24"):
        return dict(kind=kind, nx=_log(rng, 600, 20000), ny=1,
                    steps=rng.randint(64, 300) if f64 or kind[-1] == "4" else rng.randint(64, 480),
                    f64=f64, tne=tne if f64 else 0)
    if kind == "reflection":
        ny = _log(rng, 60, 300)
        return dict(kind=kind, nx=3 * ny + rng.randint(-9, 9), ny=ny, steps=rng.randint(33, 64),
                    f64=f64, tne=0)
    big = 700 if f64 else 3000 if kind == "field" else 2000
    nx, ny = _log(rng, 96, big), _log(rng, 96, big)
    # the FP32 24-velocity form loses 2e-6 a step to cancellation: short runs of it
    steps = rng.randint(4, 8) if f64 else rng.randint(9, 32) if kind == "field" else rng.randint(3, 6)
    return dict(kind=kind, nx=nx, ny=ny, steps=steps, f64=f64, tne=tne if f64 else 0,
                df32=kind == "field" and not f64 and rng.random() < 0.3,
                equal=not tne and rng.random() < 0.3)


def work(case):
    """Fields read and results written once; a state larger than the L2 cache also passes
    through memory once each way per step. Operations: what one cell's step cannot do without
    (moments, equilibrium, collision, back-transform, flux differences)."""
    cells, steps, kind = _cells(case), case["steps"], case["kind"]
    if kind == "gradient":  # forward and recomputed steps, then the reverse step
        return {"bytes": cells * 8.0 * 7, "flops": cells * steps * (2 * 400.0 + 1200.0)}
    planes = 25 if kind.endswith("24") else 17
    f64 = case.get("f64", False)
    state = cells * planes * (8.0 if f64 else 4.0)
    b = cells * 40.0 + (cells * 48.0 if f64 else state)
    if state > L2_BYTES:
        b += 2.0 * state * steps
    one_d = case.get("ny", 1) == 1
    flops = (900.0 if one_d else 1150.0) if planes == 25 else (400.0 if one_d else 550.0)
    return {"bytes": b, "flops": cells * steps * flops}


# ------------------------------------------------------------------ the inputs

def _cells(case):
    if case["kind"] == "batched":
        return int(_lengths(case, 0).sum())
    return case["nx"] * case.get("ny", 1)


def _lengths(case, seed):
    """Lengths of the instances: log-uniform, multiples of 4; the same for every seed."""
    r = np.random.default_rng(1000 * case["n"] + case["nx_max"])
    x = np.exp(r.uniform(math.log(case["nx_min"]), math.log(case["nx_max"] + 1), case["n"]))
    return np.maximum(4, (np.round(x / 4) * 4)).astype(np.int64)


def _cj(Q):
    """Chapman-Jouguet state (rho, u, T) behind a detonation into a gas with rho = p = 1."""
    q = (GAMMA * GAMMA - 1.0) * Q / GAMMA
    M2 = 1.0 + q + math.sqrt((1.0 + q) ** 2 - 1.0)
    p = (1.0 + GAMMA * M2) / (1.0 + GAMMA)
    rho = (GAMMA + 1.0) * M2 / (1.0 + GAMMA * M2)
    return rho, math.sqrt(M2 * GAMMA) * (1.0 - 1.0 / rho), p / rho


def _ripple(r, n):
    """A sum of four sine modes of 48 to 200 cells' length, at most 1 in size."""
    x = np.arange(n) / n
    s = sum(r.uniform(0.5, 1.0) * np.sin(2 * np.pi * (max(1, round(n / r.uniform(48, 200))) * x + r.uniform()))
            for _ in range(4))
    return s / np.abs(s).max()


def _modes(r, nx, ny):
    """A sum of 32 random Fourier modes (1 <= |k| <= 16) on the grid, at most 1 in size, and
    its derivatives along y and x, from per-axis tables."""
    top = max(1, min(16, min(nx, ny) // 4))
    ks = []
    while len(ks) < 32:
        k = r.integers(-top, top + 1, size=2)
        if 1 <= math.hypot(*k) <= top:
            ks.append(k)
    ks = torch.tensor(np.array(ks), dtype=F8, device=DEV)
    amp = torch.tensor(r.uniform(0, 1, 32), device=DEV)
    ph = torch.tensor(r.uniform(0, 2 * np.pi, 32), device=DEV)
    ax = 2 * np.pi * ks[:, :1] * torch.arange(nx, device=DEV, dtype=F8) / nx + ph[:, None]
    ay = 2 * np.pi * ks[:, 1:] * torch.arange(ny, device=DEV, dtype=F8) / ny
    cx, sx, cy, sy = torch.cos(ax), torch.sin(ax), torch.cos(ay), torch.sin(ay)

    def total(w, even):
        if even:
            return (cy.T * w) @ cx - (sy.T * w) @ sx
        return -((sy.T * w) @ cx + (cy.T * w) @ sx)
    phi = total(amp, True)
    return phi / phi.abs().max(), total(amp * ks[:, 1], False) / ny, total(amp * ks[:, 0], False) / nx


def _fields(case, seed):
    """rho, ux, uy, T, lambda as FP64 CUDA tensors [ny, nx]."""
    kind, r = case["kind"], np.random.default_rng([seed, 97])
    if kind in ("field", "field24"):
        # a premix with smooth random modes (5 % in rho and T, solenoidal velocities up to
        # 0.1) and a hot band above the ignition temperature: about a quarter of it reacts
        nx, ny = case["nx"], case["ny"]
        rho, T = 1.0 + 0.05 * _modes(r, nx, ny)[0], 1.0 + 0.05 * _modes(r, nx, ny)[0]
        _, dy, dx = _modes(r, nx, ny)
        peak = torch.sqrt(dx * dx + dy * dy).max()
        x = torch.arange(nx, device=DEV)
        T = T + 0.25 * ((x - int(r.integers(0, nx))) % nx < max(1, nx // 4)).to(F8)
        g = torch.Generator(device=DEV)
        g.manual_seed(int(r.integers(1 << 31)))
        lam = 0.2 * torch.rand(ny, nx, generator=g, device=DEV, dtype=F8)
        return [rho, 0.1 * dy / peak, -0.1 * dx / peak, T, lam]
    if kind == "reflection":
        # the box holds the inflow with a slight seeded disturbance
        nx, ny = case["nx"], case["ny"]
        one = torch.ones(ny, nx, dtype=F8, device=DEV)
        m = _modes(r, nx, ny)[0]
        return [one + 1e-2 * m, INFLOW[1] * one, 0.0 * one, INFLOW[3] * one, 0.0 * one]
    if kind == "batched":
        Q = _batch_rates(case, seed)[1]
        parts = []
        for n, q in zip(_lengths(case, seed), Q):
            rho, u, T = _cj(float(q))
            b = np.arange(int(n)) < 50
            parts.append(np.stack([np.where(b, rho, 1.0), np.where(b, u, 0.0), np.zeros(int(n)),
                                   np.where(b, T, 1.0), np.where(b, 1.0, 0.0)]))
        a = np.concatenate(parts, axis=1)
    else:
        nx = case["nx"]
        x = np.arange(nx)
        if kind == "sod":
            left = x < nx // 2 + int(r.integers(-nx // 20, nx // 20 + 1))
            rho = np.where(left, 1.0, 0.125 * (1 + 0.05 * r.uniform()))
            a = np.stack([rho, 0 * rho, 0 * rho, np.where(left, 1.0, 0.8), 0 * rho])
        else:
            # burnt Chapman-Jouguet gas behind the front, a quiet premix ahead of it (a wavy
            # one for the gradient, whose limiter branches are then well decided)
            b = x < (int(0.2 * nx) if kind == "detonation24" else 50) + int(r.integers(0, 40))
            rho, u, T = _cj(1.0)
            a = np.stack([np.where(b, rho, 1.0 + 0.02 * r.uniform()), np.where(b, u, 0.0), 0.0 * x,
                          np.where(b, T, 1.0 + 0.02 * r.uniform()), np.where(b, 1.0, 0.0)])
            if kind == "gradient":
                a[0] *= 1 + 2e-2 * _ripple(r, nx)
                a[3] *= 1 + 2e-2 * _ripple(r, nx)
    return [torch.tensor(v[None, :], device=DEV) for v in a]


def _rates(case, seed):
    kind, n = case["kind"], 24 if case["kind"].endswith("24") else 16
    if kind in ("field", "field24"):
        r = np.random.default_rng([seed, 98])
        return np.full(n, 5e4) if case["equal"] else r.uniform(1e4, 1e5, n)
    S = np.full(n, 1e5)
    if kind == "reflection":
        S[4:7], S[7:9] = 1.8e5, 2e5
    elif kind != "sod":
        S[4:7] = 1e4
    return S


def _batch_rates(case, seed):
    r = np.random.default_rng([seed, 99])
    a = np.exp(r.uniform(math.log(1e4), math.log(1e5), case["n"]))
    S = 10.0 * a[:, None] * np.ones((1, 16))
    S[:, 4:7] = a[:, None]
    return S, r.uniform(0.5, 2.0, case["n"])


def _params(case, seed):
    """The physical parameters of a case: plain values for the solver and for exact()."""
    kind = case["kind"]
    p = dict(gamma=GAMMA, Q=0.0, omega1=0.0, T_ig=1.1, dx=1e-3, dt=1e-5, bc=(1, 0),
             S=_rates(case, seed) if kind != "batched" else None)
    if kind in ("field", "field24"):
        p.update(Q=1.0, omega1=2e4, dt=5e-6, bc=(0, 0))
    elif kind == "reflection":
        p.update(gamma=1.5, dt=5e-6, bc=(5, 5))
    elif kind == "detonation24":
        p.update(Q=1.0, omega1=1e3, dx=2e-4, dt=5e-6)
    elif kind == "batched":
        p.update(Q=1.0, omega1=2e4, dx=1e-4, dt=1e-6)
    elif kind != "sod":
        p.update(Q=1.0, omega1=2e4, dx=1e-4, dt=2e-6)
    return p


def _target(case, seed):
    r = np.random.default_rng([seed, 96])
    return 1.0 + 0.05 * _ripple(r, case["nx"])


def prepare(case, seed):
    kind, p = case["kind"], _params(case, seed)
    fields = _fields(case, seed)
    kw = dict(gamma=p["gamma"], T_ig=p["T_ig"], dx=p["dx"], dy=p["dx"], dt=p["dt"])
    if kind == "batched":
        S, Q = _batch_rates(case, seed)
        s = lbkm.Solver.batched(_lengths(case, seed), inst_S=S, inst_Q=Q, omega1=p["omega1"], **kw)
        fields = [f.reshape(1, -1) for f in fields]
        s.init_fields(*fields)
        s.autotune(3)
    else:
        kw.update(nx=case["nx"], ny=case.get("ny", 1), S=p["S"], Q=p["Q"], omega1=p["omega1"],
                  bc=p["bc"], precision=lbkm.F64 if case.get("f64", True) else lbkm.F32,
                  tne_every=case.get("tne", 0), tne_capacity=case["steps"])
        if kind.endswith("24"):
            s = lbkm.Solver24(v=SETS24[0], eta=SETS24[1], **kw)
        else:
            if kind == "reflection":
                def side(code, st):
                    return (code, st[0], st[1], st[2], st[3], 0.0)
                kw.update(orbit_speed=[o[0] for o in ORBITS16_REFLECTION],
                          orbit_eta=[o[1] for o in ORBITS16_REFLECTION],
                          sides=(side(3, INFLOW), side(1, INFLOW), side(4, INFLOW), side(3, LID)))
            if case.get("df32"):
                kw.update(recovery=lbkm.RECOVER_DF32)
            s = lbkm.Solver(**kw)
    return dict(solver=s, fields=fields, steps=case["steps"], tne=case.get("tne", 0),
                target=_target(case, seed) if kind == "gradient" else None)


def run(state):
    s = state["solver"]
    s.init_fields(*state["fields"])
    if state["target"] is not None:
        return s.grad(state["target"], state["steps"], checkpoint_every=64)
    s.step(state["steps"])
    f64 = s.params.precision == lbkm.F64
    out = {}
    if not f64:
        out["planes"] = s.planes_device()
    elif s.ny > 1:
        out["macros"] = s.macros(device=True)
    else:  # a plane run: no transverse velocity is asked for
        out["macros"] = s.macros(device=True, out={k: torch.empty(1, s.nx, dtype=F8, device=DEV)
                                                   for k in ("rho", "ux", "T", "p", "lam")})
    if state["tne"]:
        rec = s.tne_history()
        # the records of an FP32 run are kept in its own precision
        out["tne"] = {k: np.array([x[k] for x in rec], np.float64 if f64 else np.float32)
                      for k in ("sum", "abs_sum", "min", "max", "d_sum", "d2_sum")}
    return out


# ------------------------------------------------------------------ the model in 64 bits

class _Model:
    def __init__(self, case, seed, p):
        self.kind, self.p = case["kind"], p
        self.n24 = self.kind.endswith("24")
        if self.n24:
            orbits = [(v, e) for v, e in zip(*SETS24) for _ in (0, 1)]
        else:
            orbits = ORBITS16_REFLECTION if self.kind == "reflection" else ORBITS16
        unit = (((1, 0), (0, 1), (-1, 0), (0, -1)), ((1, 1), (-1, 1), (-1, -1), (1, -1)))
        v = [(c * a, c * b, e) for o, (c, e) in enumerate(orbits) for a, b in unit[o % 2]]
        self.vx, self.vy, self.eta = (torch.tensor([t[k] for t in v], dtype=F8, device=DEV)
                                      for k in range(3))
        self.flip = [next(j for j in range(len(v)) if j // 4 == i // 4 and v[j][0] == v[i][0]
                          and v[j][1] == -v[i][1]) for i in range(len(v))]
        a, b, e2 = self.vx, self.vy, self.eta ** 2
        v2, w = a * a + b * b, a * a + b * b + e2
        rows = [torch.ones_like(a), a, b, w, a * a, a * b, b * b, w * a, w * b, a ** 3, a * a * b,
                a * b * b, b ** 3, w * a * a, w * a * b, w * b * b]
        if self.n24:
            rows += [e2 * a * a, e2 * a * b, e2 * b * b, w * e2, w * v2 * a, w * v2 * b,
                     w * e2 * a, w * e2 * b]
        self.M = torch.stack(rows)
        self.Minv = torch.linalg.inv(self.M.cpu()).to(DEV)
        self.I = 2.0 / (p["gamma"] - 1.0) - 2.0
        self.DI = 2.0 + self.I
        self.S, self.Q, self.omega1 = p["S"], p["Q"], p["omega1"]
        self.lengths = _lengths(case, seed) if self.kind == "batched" else None
        if self.lengths is not None:
            n = torch.tensor(self.lengths, device=DEV)
            first = torch.cumsum(n, 0) - n
            lo, hi = torch.repeat_interleave(first, n), torch.repeat_interleave(first + n - 1, n)
            at = torch.arange(int(n.sum()), device=DEV)
            self.index = {d: torch.minimum(torch.maximum(at + d, lo), hi) for d in (-2, -1, 1, 2)}
        self.side = None
        if self.kind == "reflection":
            self.side = [self.start(*(torch.full((1,), x, dtype=F8, device=DEV) for x in
                                      (s[0], s[1], s[2], s[3]))) for s in (INFLOW, LID)]

    def mul(self, A, x):
        return (A @ x.reshape(x.shape[0], -1)).reshape(A.shape[0], *x.shape[1:])

    def feq(self, rho, ux, uy, T):
        DI, I = self.DI, self.I
        u2 = ux * ux + uy * uy
        A, B = (DI + 2) * T + u2, (DI + 4) * T + u2
        q = [rho, rho * ux, rho * uy, rho * (DI * T + u2), rho * (T + ux * ux), rho * ux * uy,
             rho * (T + uy * uy), rho * ux * A, rho * uy * A, rho * ux * (3 * T + ux * ux),
             rho * uy * (T + ux * ux), rho * ux * (T + uy * uy), rho * uy * (3 * T + uy * uy),
             rho * (A * T + ux * ux * B), rho * ux * uy * B, rho * (A * T + uy * uy * B)]
        if self.n24:
            C = u2 * u2 + 4 * (DI + 4) * T * T + (DI + 10) * u2 * T
            q += [rho * I * T * (T + ux * ux), rho * ux * uy * I * T, rho * I * T * (T + uy * uy),
                  rho * I * T * (u2 + (2 + 3 * I) * T), rho * ux * C, rho * uy * C,
                  rho * ux * I * T * (u2 + (4 + 3 * I) * T), rho * uy * I * T * (u2 + (4 + 3 * I) * T)]
        return torch.stack(q)

    def dfeq(self, rho, ux, uy, T):
        DI = self.DI
        u2, z = ux * ux + uy * uy, torch.zeros_like(rho)
        dA = 2 * (DI + 2) * T + u2
        return torch.stack([z, z, z, rho * DI, rho, z, rho, rho * ux * (DI + 2),
                            rho * uy * (DI + 2), 3 * rho * ux, rho * uy, rho * ux, 3 * rho * uy,
                            rho * (dA + ux * ux * (DI + 4)), rho * ux * uy * (DI + 4),
                            rho * (dA + uy * uy * (DI + 4))])

    def start(self, rho, ux, uy, T):
        return self.mul(self.Minv, self.feq(rho, ux, uy, T))

    def macros(self, f):
        rho, jx, jy, e = self.mul(self.M[:4], f)
        ux, uy = jx / rho, jy / rho
        return rho, ux, uy, (e / rho - ux * ux - uy * uy) / self.DI

    def shift(self, f, d, axis, scalar=None):
        """f (or one plane of it, `scalar` naming what it is) at the cell d away along x
        (axis -1) or y (axis -2), beyond the edge as the side's condition has it."""
        if self.lengths is not None:
            return f[..., self.index[d]]
        n, bc = f.shape[axis], self.p["bc"][0 if axis == -1 else 1]
        if bc == 0:
            return torch.roll(f, -d, axis)
        at = torch.arange(n, device=DEV) + d
        g = f.index_select(f.dim() + axis, at.clamp(0, n - 1))
        if bc == 5:
            k, out = abs(d), slice(0, abs(d)) if d < 0 else slice(n - abs(d), n)
            place = (Ellipsis, out) if axis == -1 else (Ellipsis, out, slice(None))
            if axis == -1 and d < 0:
                g[place] = self.ghost(0, scalar, f.dim())
            elif axis == -2 and d > 0:
                g[place] = self.ghost(1, scalar, f.dim())
            elif axis == -2:  # the reflecting floor: rows k-1 .. 0, v_y reversed
                m = f[..., :k, :].flip(-2)
                g[place] = m[self.flip] if scalar is None else (-m if scalar == "uy" else m)
        return g

    def ghost(self, side, scalar, dim):
        if scalar is None:
            return self.side[side].reshape(-1, *([1] * (dim - 1)))
        st = (INFLOW, LID)[side]
        return {"ux": st[1], "uy": st[2], "lam": 0.0}[scalar]

    @staticmethod
    def mm(a, b):
        return torch.where(a * b > 0, torch.where(a.abs() <= b.abs(), a, b), torch.zeros_like(a))

    def nnd(self, f, axis, scalar=None):
        """(upwind differences for v > 0, for v < 0) along one axis."""
        g = {d: self.shift(f, d, axis, scalar) for d in (-2, -1, 1, 2)}
        d0, d1, d2, d3 = g[-1] - g[-2], f - g[-1], g[1] - f, g[2] - g[1]
        m1, m2, m3 = self.mm(d0, d1), self.mm(d1, d2), self.mm(d2, d3)
        return d1 + 0.5 * (m2 - m1), d2 - 0.5 * (m3 - m2)

    def step(self, f, lam):
        p, dt, dx = self.p, self.p["dt"], self.p["dx"]
        two = f.shape[1] > 1
        nd = (1,) * (f.dim() - 1)
        rho, ux, uy, T = self.macros(f)
        q = self.feq(rho, ux, uy, T)
        D = self.mul(self.M, f)[4:] - q[4:]
        S = self.S if torch.is_tensor(self.S) else torch.as_tensor(self.S, dtype=F8, device=DEV)
        S = S.reshape(-1, *nd) if S.dim() == 1 else S

        def grad(u, axis, name):
            return (self.shift(u, 1, axis, name) - self.shift(u, -1, axis, name)) / (2 * dx)
        gxx, gyx = grad(ux, -1, "ux"), grad(uy, -1, "uy")
        z = torch.zeros_like(rho)
        gxy, gyy = (grad(ux, -2, "ux"), grad(uy, -2, "uy")) if two else (z, z)
        th, sh = (gxx + gyy) / self.DI, gyx + gxy
        A8 = rho * T * (1 - S[7] / S[4]) * (4 * ux * (gxx - th) + 2 * uy * sh)
        A9 = rho * T * (1 - S[8] / S[6]) * (4 * uy * (gyy - th) + 2 * ux * sh)
        dl = torch.where(T > p["T_ig"], (1 - lam) * -torch.expm1(-self.omega1 * rho * T * dt), z)
        om = -S[4:] * D
        om = torch.cat([z[None], z[None], z[None], z[None], om[:3], (om[3] + A8)[None],
                        (om[4] + A9)[None], om[5:]])
        if self.n24:
            fe = self.mul(self.Minv, q)
            c2 = (self.vx.reshape(-1, *nd) - ux) ** 2 + (self.vy.reshape(-1, *nd) - uy) ** 2
            I = self.I
            om = self.mul(self.Minv, om) + fe * (self.Q * dl / dt / (I * self.DI * T * T)) * (
                -3 * I * T + I * c2 + (self.eta ** 2).reshape(-1, *nd))
            del fe, c2
        else:
            om = self.mul(self.Minv, om + self.dfeq(rho, ux, uy, T) * (2 * self.Q * dl / (self.DI * dt)))
        up, un = self.nnd(f, -1)
        vx, vy = self.vx.reshape(-1, *nd), self.vy.reshape(-1, *nd)
        adv = (vx.clamp(min=0) * up + vx.clamp(max=0) * un) / dx
        lp, ln = self.nnd(lam, -1, "lam")
        la = torch.where(ux > 0, ux * lp, torch.where(ux < 0, ux * ln, z)) / dx
        if two:
            up, un = self.nnd(f, -2)
            adv = adv + (vy.clamp(min=0) * up + vy.clamp(max=0) * un) / dx
            lp, ln = self.nnd(lam, -2, "lam")
            la = la + torch.where(uy > 0, uy * lp, torch.where(uy < 0, uy * ln, z)) / dx
        return f + dt * (om - adv), (lam - dt * la + dl).clamp(0.0, 1.0), D


def _record(D, area):
    """The TNE record of one step's Delta_5.. (sums weighted by the cell area)."""
    flat = D.reshape(D.shape[0], -1)
    four = torch.zeros(4, dtype=F8, device=DEV)
    d2 = (flat * flat).sum(0)
    rec = {"sum": flat.sum(1) * area, "abs_sum": flat.abs().sum(1) * area,
           "min": flat.min(1).values, "max": flat.max(1).values}
    rec = {k: torch.cat([four, v]).cpu().numpy() for k, v in rec.items()}
    return rec | {"d_sum": float(d2.sqrt().sum()) * area, "d2_sum": float(d2.sum()) * area}


def _gradient(case, seed, m, fields):
    """J and its derivatives by reverse-mode differentiation, segments of 64 steps recomputed."""
    from torch.utils.checkpoint import checkpoint
    p = m.p
    rho0 = fields[0].clone().requires_grad_()
    m.S = torch.tensor(p["S"], device=DEV, requires_grad=True)
    m.Q = torch.tensor(p["Q"], dtype=F8, device=DEV, requires_grad=True)
    m.omega1 = torch.tensor(p["omega1"], dtype=F8, device=DEV, requires_grad=True)

    def segment(f, lam, S, Q, omega1, n):
        t = torch.zeros((), dtype=F8, device=DEV)
        for _ in range(n):
            f, lam, D = m.step(f, lam)
            t = t + (D * D).sum() * p["dx"] * p["dt"]
        return f, lam, t
    f, lam = m.start(rho0, fields[1], fields[2], fields[3]), fields[4]
    jt = torch.zeros((), dtype=F8, device=DEV)
    for k in range(0, case["steps"], 32):
        f, lam, t = checkpoint(segment, f, lam, m.S, m.Q, m.omega1, min(32, case["steps"] - k),
                               use_reentrant=False)
        jt = jt + t
    rho = m.mul(m.M[:1], f)[0]
    jm = 0.5 * ((rho - torch.tensor(_target(case, seed), device=DEV)) ** 2).sum() * p["dx"]
    (jm + jt).backward()
    dS = m.S.grad.clone()
    dS[:4] = 0.0
    return {"J": float(jm + jt), "J_mismatch": float(jm), "J_tne": float(jt),
            "dS": dS.cpu().numpy(), "dQ": float(m.Q.grad), "domega1": float(m.omega1.grad),
            "domega2": None, "drho0": rho0.grad.reshape(-1).cpu().numpy(), "df0": None}


def exact(case, seed):
    p = _params(case, seed)
    fields = _fields(case, seed)
    m = _Model(case, seed, p)
    if case["kind"] == "gradient":
        return _gradient(case, seed, m, fields)
    with torch.no_grad():
        if case["kind"] == "batched":
            S, Q = _batch_rates(case, seed)
            per = torch.tensor(_lengths(case, seed), device=DEV)
            m.S = torch.repeat_interleave(torch.tensor(S.T.copy(), device=DEV), per, 1)[:, None, :]
            m.Q = torch.repeat_interleave(torch.tensor(Q, device=DEV), per)[None, :]
        rho, ux, uy, T, lam = fields
        f = m.start(rho, ux, uy, T)
        recs = []
        for _ in range(case["steps"]):
            g, lam, D = m.step(f, lam)
            f = g
            if case.get("tne"):
                recs.append(_record(D, p["dx"] * p["dx"]))
        if case.get("f64", False):
            rho, ux, uy, T = m.macros(f)
            out = {"macros": dict(rho=rho, ux=ux, T=T, p=rho * T, lam=lam)}
            if f.shape[1] > 1:
                out["macros"]["uy"] = uy
        else:
            out = {"planes": torch.cat([f, lam[None]])}
    if case.get("tne"):
        out["tne"] = {k: np.array([x[k] for x in recs]) for k in recs[0]}
    return out
