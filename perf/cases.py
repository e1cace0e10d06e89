"""The work that users of the solver have it do, as cases to be timed.

A case is a dict of plain values; its ``kind`` is one of

  tube      a whole run of a shock tube on D2Q9: initial fields in, n steps, fields out
  vortex    n steps of a shock-vortex interaction on D2Q9 (zero-gradient ends, or a fixed inflow)
  sheet     n steps of decaying two-dimensional turbulence on a periodic D2Q9 sheet
  box       n steps of decaying compressible turbulence on a periodic D3Q27 box
  history   the same with the turbulence statistics of the state reached (one sample of K(t), theta_rms(t))
  inplace   n steps of such a box on the single-store layout, for boxes that two stores would not leave room for
  embedded  n allocation-free steps on stores that the caller owns
  snapshot  fields, conserved totals and statistics of a state, as a run writes them out
  ensemble  n steps of a batch of uneven shock tubes and shock-vortex cases

Step counts are even, so that the state is back in the first store after every pass.
Inputs come from the seed alone; ``exact`` repeats a pass in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2102_09512_gb300 import elbm as E

DEV = "cuda"
F64 = torch.float64
GAMMA, T0 = 1.4, 0.15
VALUE = {"f64": (8, torch.float64), "f32": (4, torch.float32), "f16dev": (2, torch.float16), "bf16dev": (2, torch.bfloat16)}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the shock tube of the validation runs: 3,200 nodes, all launches and latency
        dict(name="tube_f64_800x4", kind="tube", store="f64", nx=800, ny=4, steps=500),
        # the shock-vortex run at the paper's size, supersonic inflow, double precision
        dict(name="vortex_f64_1680x1440", kind="vortex", store="f64", nx=1680, ny=1440, inflow=True, steps=4),
        # the configured shock-vortex run, single precision
        dict(name="vortex_f32_1024sq", kind="vortex", store="f32", nx=1024, ny=1024, inflow=False, steps=20),
        # a large two-dimensional flow with the 16-bit store
        dict(name="sheet_f16_4096sq", kind="sheet", store="f16dev", nx=4096, ny=4096, steps=8),
        # the batched sweep of 64 lattices between 256^2 and 1024^2
        dict(name="ensemble_f32_64", kind="ensemble", store="f32", count=64, side_min=256, side_max=1024, steps=8),
        # the headline box in both storage widths
        dict(name="box_f32_256cube", kind="box", store="f32", nx=256, ny=256, nz=256, steps=10),
        dict(name="box_f16_256cube", kind="box", store="f16dev", nx=256, ny=256, nz=256, steps=10),
        # the double-precision run that reduced stores are compared with
        dict(name="box_f64_128cube", kind="box", store="f64", nx=128, ny=128, nz=128, steps=2),
        # the configured 128^3 run with its histories
        dict(name="history_f32_128cube", kind="history", store="f32", nx=128, ny=128, nz=128, steps=20),
        # the single store, as grids that fill the device use it
        dict(name="inplace_f32_320cube", kind="inplace", store="f32", nx=320, ny=320, nz=320, steps=4),
        # a solver embedded in another application, small and ragged
        dict(name="embedded_f32_61x45x53", kind="embedded", store="f32", nx=61, ny=45, nz=53, steps=16),
        # what a run writes out now and then
        dict(name="snapshot_f32_256cube", kind="snapshot", store="f32", nx=256, ny=256, nz=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _store(rng):
    return rng.choice(["f64", "f32", "f32", "f16dev", "f16dev", "bf16dev"])


def draw(rng):
    kind = rng.choice(["tube", "vortex", "sheet", "box", "box", "history", "inplace", "embedded", "snapshot", "ensemble"])
    if kind == "tube":
        return dict(kind=kind, store=rng.choice(["f64", "f64", "f32"]), nx=_log(rng, 200, 2000), ny=rng.randint(1, 8), steps=2 * rng.randint(50, 250))
    if kind == "vortex":
        return dict(kind=kind, store=rng.choice(["f64", "f32"]), nx=_log(rng, 256, 2000), ny=_log(rng, 200, 1600), inflow=rng.random() < 0.5, steps=2 * rng.randint(1, 3))
    if kind == "sheet":
        store = _store(rng)
        hi = 1600 if store == "f64" else 3600
        return dict(kind=kind, store=store, nx=_log(rng, 96, hi), ny=_log(rng, 96, hi), steps=2 * rng.randint(1, 4))
    if kind == "ensemble":
        lo = rng.randint(96, 400)
        return dict(kind=kind, store=rng.choice(["f32", "f32", "f16dev"]), count=rng.randint(3, 40), side_min=lo, side_max=lo + rng.randint(30, 500), steps=2 * rng.randint(1, 6))
    c = dict(kind=kind, store="f32" if kind == "history" else _store(rng))
    hi = 100 if kind == "embedded" else 150 if c["store"] == "f64" else 240
    for axis in ("nx", "ny", "nz"):
        c[axis] = _log(rng, 24, hi)
    if kind == "embedded" and c["store"] == "f64":   # the static scratch holds 0.69 million nodes of this store
        c["nz"] = min(c["nz"], 600_000 // (c["nx"] * c["ny"]))
    if kind != "snapshot":
        c["steps"] = 2 * rng.randint(1, 2 if c["store"] == "f64" else 5)
    return c


def nodes(case):
    if case["kind"] == "ensemble":
        # the sides are uniform in [side_min, side_max]: their mean square
        lo, hi = case["side_min"], case["side_max"]
        return case["count"] * (lo * lo + lo * hi + hi * hi) / 3.0
    return case["nx"] * case["ny"] * case.get("nz", 1)


def work(case):
    """Bytes: the populations of every node read and written once a step, a snapshot's read once and its fields
    written.  Operations: those of the update as the paper writes it, about 510 (D3Q27) and 190 (D2Q9) a node."""
    Q = 9 if case["kind"] in ("tube", "vortex", "sheet", "ensemble") else 27
    N, pair = nodes(case), 2 * VALUE[case["store"]][0]
    if case["kind"] == "snapshot":
        return {"bytes": N * (Q * pair + 5 * 8), "flops": N * 250}
    fields = 8.0 * N * 4 * 2 if case["kind"] == "tube" else 0.0
    return {"bytes": N * case["steps"] * 2 * Q * pair + fields, "flops": N * case["steps"] * (510 if Q == 27 else 190)}


# ---------------------------------------------------------------------------
# initial fields, on the device in FP64: rho (nz, ny, nx), u (D, nz, ny, nx), T
# ---------------------------------------------------------------------------
def _noise(shape, k0, gen):
    """A real field of unit variance with the shell spectrum k^4 exp(-2 (k/k0)^2) (wavenumbers of the longest axis)."""
    n = max(shape)
    k = [torch.fft.fftfreq(m, 1.0 / n, device=DEV, dtype=F64) for m in shape[:-1]]
    k.append(torch.fft.rfftfreq(shape[-1], 1.0 / n, device=DEV, dtype=F64))
    k2 = sum(g * g for g in torch.meshgrid(*k, indexing="ij"))
    w = torch.fft.rfftn(torch.randn(shape, generator=gen, device=DEV, dtype=F64))
    w *= torch.sqrt(k2) * torch.exp(-k2 / (k0 * k0))
    f = torch.fft.irfftn(w, s=shape)
    f -= f.mean()
    return f / torch.sqrt((f * f).mean()).clamp_min(1e-30)


def _turbulence(case, seed):
    """Turbulent velocity of Mach number 0.12 (solenoidal in 3D, on a sheet from a stream function) with density and
    temperature fluctuations, carried along by a mean flow (a component that changes sign flips the upwind side at
    nodes where it is a rounding error away from zero); the viscosity keeps Re_lambda = 72 (at least 0.005)."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    D = 3 if "nz" in case else 2
    shape = (case.get("nz", 1), case["ny"], case["nx"])
    fft_shape = shape if D == 3 else shape[1:]
    n = max(shape)
    k0 = min(4.0 if D == 3 else 8.0, n / 16.0)

    def diff(a, axis):
        return 0.5 * (torch.roll(a, -1, axis) - torch.roll(a, 1, axis))

    psi = [_noise(fft_shape, k0, gen).reshape(shape) for _ in range(3 if D == 3 else 1)]
    u = torch.empty((D,) + shape, device=DEV, dtype=F64)
    if D == 3:   # curl of a vector potential; axes are (z, y, x)
        u[0] = diff(psi[2], 1) - diff(psi[1], 0)
        u[1] = diff(psi[0], 0) - diff(psi[2], 2)
        u[2] = diff(psi[1], 2) - diff(psi[0], 1)
    else:
        u[0] = diff(psi[0], 1)
        u[1] = -diff(psi[0], 2)
    u *= 0.12 * math.sqrt(GAMMA * T0) / torch.sqrt((u * u).sum(0).mean()).clamp_min(1e-30)
    dux = diff(u[0], 2)
    lam = torch.sqrt((u[0] ** 2).mean() / (dux * dux).mean().clamp_min(1e-30))
    mu0 = max(0.005, float(torch.sqrt((u * u).mean()) * lam) / 72.0)
    u += torch.tensor([0.1, 0.09, 0.09][:D], device=DEV, dtype=F64).reshape(D, 1, 1, 1)
    rho = 1.0 + 0.02 * _noise(fft_shape, k0, gen).reshape(shape)
    T = T0 * (1.0 + 0.01 * _noise(fft_shape, k0, gen).reshape(shape))
    return dict(D=D, nx=case["nx"], ny=case["ny"], nz=shape[0], rho=rho, u=u, T=T, Pr=0.7, mu0=mu0, mu_exp=0.76,
                bc=(0,) * 6, fixed=(0.0,) * 5, T_scale=T0)


def _tube(nx, ny, gen):
    """A shock tube of pressure ratio about 10 with its membrane near the middle and zero-gradient ends, in a gas that
    drifts to the right: where the gas ahead of a shock is at rest, the last bit of a sum decides the upwind side."""
    a = torch.rand(4, generator=gen, dtype=F64).tolist()
    xm = int(nx * (0.45 + 0.1 * a[0]))
    left = (torch.arange(nx, device=DEV) < xm).expand(1, ny, nx)
    rho = torch.where(left, 1.0, 0.125 + 0.025 * a[1]).to(F64)
    T = torch.where(left, 0.15, 0.12 + 0.004 * a[2]).to(F64)
    u = torch.zeros((2, 1, ny, nx), device=DEV, dtype=F64)
    u[0] = 0.04 + 0.02 * a[3]
    return dict(D=2, nx=nx, ny=ny, nz=1, rho=rho, u=u, T=T, Pr=0.71, mu0=0.015, mu_exp=0.0, bc=(1, 1, 0, 0, 0, 0), fixed=(0.0,) * 5,
                T_scale=0.15)


def _vortex(nx, ny, inflow, gen, mach=(1.18, 1.22)):
    """A standing normal shock and an isentropic vortex of Mach number 0.25 upstream of it."""
    a = torch.rand(2, generator=gen, dtype=F64).tolist()
    Ma, Mv, Tl = mach[0] + (mach[1] - mach[0]) * a[0], 0.25, 0.05
    r_v = min(nx, ny) / 32.0 if nx != 1680 else 60.0
    c = math.sqrt(GAMMA * Tl)
    M2 = Ma * Ma
    r = (GAMMA + 1.0) * M2 / ((GAMMA - 1.0) * M2 + 2.0)
    pr = 1.0 + 2.0 * GAMMA / (GAMMA + 1.0) * (M2 - 1.0)
    x = torch.arange(nx, device=DEV, dtype=F64)[None, :]
    y = torch.arange(ny, device=DEV, dtype=F64)[:, None]
    left = (x < 8.0 * r_v).expand(ny, nx)
    one = torch.ones((ny, nx), device=DEV, dtype=F64)
    rho_b, P_b, ux_b = torch.where(left, one, one * r), torch.where(left, one * Tl, one * Tl * pr), torch.where(left, one * Ma * c, one * Ma * c / r)
    xv, yv = 6.0 * r_v, ny / 2.0 + r_v * (a[1] - 0.5)
    r2 = ((x - xv) ** 2 + (y - yv) ** 2) / (r_v * r_v)
    base = 1.0 - 0.5 * (GAMMA - 1.0) * Mv * Mv * torch.exp(1.0 - r2)
    rho = rho_b * base ** (1.0 / (GAMMA - 1.0))
    T = P_b * base ** (GAMMA / (GAMMA - 1.0)) / rho
    amp = c * Mv * torch.exp(0.5 * (1.0 - r2))
    u = torch.stack([ux_b + amp * (y - yv) / r_v, -amp * (x - xv) / r_v])[:, None]
    return dict(D=2, nx=nx, ny=ny, nz=1, rho=rho[None], u=u, T=T[None], Pr=0.75, mu0=c * 60.0 / 800.0, mu_exp=0.0,
                bc=(2 if inflow else 1, 1, 0, 0, 0, 0), fixed=(1.0, Ma * c, 0.0, 0.0, Tl), T_scale=Tl)


def _members(case, seed):
    """The lattices of an ensemble: square, sides uniform in the case's range (on a fixed grid of sizes, as a sweep has
    them; the sizes belong to the case, the states to the seed), shock tubes and shock-vortex cases in turn."""
    sides = np.random.default_rng(7).uniform(case["side_min"], case["side_max"], case["count"]).round().astype(int)
    gen = torch.Generator()
    gen.manual_seed(seed)
    for k, s in enumerate(sides):
        yield _tube(int(s), int(s), gen) if k % 2 == 0 else _vortex(int(s), int(s), False, gen, (1.1, 1.5))


def _problem(case, seed):
    gen = torch.Generator()
    gen.manual_seed(seed)
    if case["kind"] == "tube":
        return _tube(case["nx"], case["ny"], gen)
    if case["kind"] == "vortex":
        return _vortex(case["nx"], case["ny"], case["inflow"], gen)
    return _turbulence(case, seed)


def _params(q, store):
    return E.make_params(q["D"], q["nx"], q["ny"], q["nz"], GAMMA, q["Pr"], q["mu0"], q["T_scale"], q["mu_exp"], q["bc"],
                         store, 0, 1.0, q["T_scale"], q["fixed"])


# ---------------------------------------------------------------------------
# a user's program
# ---------------------------------------------------------------------------
class State:
    pass


def prepare(case, seed):
    s = State()
    s.case, s.kind, s.steps = case, case["kind"], case.get("steps", 0)
    dtype = VALUE[case["store"]][1]
    if s.kind == "ensemble":
        members = list(_members(case, seed))
        s.ens = E.Ensemble([_params(q, case["store"]) for q in members])
        for k, q in enumerate(members):
            s.ens.set_fields(k, q["rho"].cpu().numpy(), q["u"].cpu().numpy(), q["T"].cpu().numpy())
        s.ens.tune(use_cache=True)
        s.out = s.ens.pop_a.view(dtype)
        return s
    q = _problem(case, seed)
    p = _params(q, case["store"])
    s.solver = E.Solver(p, layout=E.ELBM_LAYOUT_AA if s.kind == "inplace" else E.ELBM_LAYOUT_PINGPONG)
    rho, u, T = (q[k].reshape(-1).contiguous() for k in ("rho", "u", "T"))
    s.solver.set_fields(rho, u, T)
    if s.kind == "tube":
        s.fields = rho, u, T
        s.result = torch.empty_like(rho), torch.empty_like(u), torch.empty_like(T)
    elif s.kind == "snapshot":
        s.result = torch.empty_like(rho), torch.empty_like(u), torch.empty_like(T)
        s.snap = [t.to(torch.float32) for t in s.result]   # single-precision files
    else:
        s.out = s.solver.pop_a.view(dtype)
    if s.kind == "embedded":
        s.params, s.pops = p, (s.solver.pop_a.data_ptr(), s.solver.pop_b.data_ptr())
    torch.cuda.synchronize()
    return s


def run(s):
    if s.kind == "ensemble":
        s.ens.step(s.steps)
        return s.out
    if s.kind == "tube":
        s.solver.set_fields(*s.fields)
        s.solver.step(s.steps)
        s.solver.fields_device(*s.result)
        return s.result if s.case["store"] == "f64" else tuple(t.to(torch.float32) for t in s.result)
    if s.kind == "snapshot":
        s.solver.fields_device(*s.result)
        for a, b in zip(s.snap, s.result):
            a.copy_(b)
        # a history file holds single precision too
        return s.snap, np.asarray(s.solver.conservation(), np.float32), _stats(s.solver)
    if s.kind == "embedded":
        stream = s.solver.stream.cuda_stream
        a, b = s.pops
        for _ in range(s.steps // 2):
            for src, dst in ((a, b), (b, a)):
                if E.elbm_step_noalloc(s.params, src, dst, stream) != E.ELBM_OK:
                    raise RuntimeError("elbm_step_noalloc failed")
        return s.out
    s.solver.step(s.steps)
    if s.kind == "history":
        return s.out, _stats(s.solver)
    return s.out


# Statistics of a history: the mean values and those of the gradients (the rms values of rho and T are differences of nearly
# equal sums).
STATS = ("rho_mean", "K", "u_rms", "theta_rms", "T_mean", "dudx2", "omega_rms", "enstrophy", "dissipation", "lambda", "Re_lambda",
         "rho_rms", "T_rms")


def _stats(solver):
    d = solver.turbulence_stats()
    return np.asarray([d[k] for k in STATS], np.float32)


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch: the paper's equations on whole fields
# ---------------------------------------------------------------------------
def _psi(xi, P):
    return [0.5 * (P - xi), 1.0 - P, 0.5 * (P + xi)]


def _gpsi(u, T):
    """Psi_c(O, O^2) applied to u^2/2."""
    o = T * u + 0.5 * u ** 3
    s = T * T + 2.5 * T * u * u + 0.5 * u ** 4
    return [0.5 * (s - o), 0.5 * u * u - s, 0.5 * (s + o)]


class Exact:
    """State arrays f, g of shape (Q, nz, ny, nx); direction i = a + 3 b + 9 c has velocity (a - 1, b - 1, c - 1)."""

    def __init__(self, q):
        self.q, self.D = q, q["D"]
        self.Q = 27 if self.D == 3 else 9
        self.c = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1 if self.D == 3 else 0) for i in range(self.Q)]
        rho, u, T = q["rho"], q["u"], q["T"]
        self.f, self.g = self.equilibrium(rho, u, T)
        if 2 in q["bc"]:
            r, *v, t = (torch.tensor(x, device=DEV, dtype=F64) for x in q["fixed"])
            self.ghost_f, self.ghost_g = self.equilibrium(r, torch.stack(v[:self.D]), t)
            self.ghost_Q = [r * v[a] * (1.0 - 3.0 * t - v[a] ** 2) for a in range(self.D)]
        self.collide()

    def factors(self, u, T, extra=None):
        z = torch.zeros_like(T)
        P = [T + u[a] ** 2 + (extra[a] if extra is not None else 0.0) for a in range(self.D)]
        phi = [_psi(u[a], P[a]) for a in range(self.D)]
        return phi + [[z, torch.ones_like(T), z]] * (3 - self.D)

    def equilibrium(self, rho, u, T):
        X = self.factors(u, T)
        S = [_gpsi(u[a], T) for a in range(self.D)] + [[torch.zeros_like(T)] * 3] * (3 - self.D)
        f, g = (torch.empty((self.Q,) + T.shape, device=DEV, dtype=F64) for _ in range(2))
        for i, c in enumerate(self.c):
            f[i], g[i] = self.f_dir(c, rho, X), self.g_dir(c, rho, T, X, S)
        return f, g

    @staticmethod
    def f_dir(c, rho, X):
        return rho * X[0][c[0] + 1] * X[1][c[1] + 1] * X[2][c[2] + 1]

    @staticmethod
    def g_dir(c, rho, T, X, S):
        x, y, z = (X[a][c[a] + 1] for a in range(3))
        sx, sy, sz = (S[a][c[a] + 1] for a in range(3))
        return rho * ((T / (GAMMA - 1.0) * x + sx) * y * z + x * (sy * z + y * sz))

    def shifted(self, a, axis, d):
        """Values at x - d e_axis: periodic, or the nearest node of the grid.  axis 0 is x (the last dimension)."""
        dim = a.dim() - 1 - axis
        out = torch.roll(a, d, dim)
        if d and self.q["bc"][2 * axis] != 0:
            n = a.shape[dim]
            out.narrow(dim, 0 if d > 0 else n - 1, 1).copy_(a.narrow(dim, 0 if d > 0 else n - 1, 1))
        return out

    def stream(self):
        for h, ghost in ((self.f, "ghost_f"), (self.g, "ghost_g")):
            for i, c in enumerate(self.c):
                v = h[i]
                for axis in range(self.D):
                    if c[axis]:
                        v = self.shifted(v, axis, c[axis])
                if 2 in self.q["bc"]:
                    for axis in range(self.D):
                        for side in (0, 1):
                            if self.q["bc"][2 * axis + side] == 2 and c[axis] == (1 if side == 0 else -1):
                                dim = v.dim() - 1 - axis
                                v.narrow(dim, 0 if side == 0 else v.shape[dim] - 1, 1).fill_(getattr(self, ghost)[i])
                h[i] = v

    def moments(self):
        rho, E_ = self.f.sum(0), self.g.sum(0)
        j = [sum(c[a] * self.f[i] for i, c in enumerate(self.c) if c[a]) for a in range(self.D)]
        u = [x / rho for x in j]
        T = (GAMMA - 1.0) * (E_ / rho - 0.5 * sum(x * x for x in u))
        return rho, u, T

    def gradient(self, Qa, ua, axis):
        lo, hi = self.shifted(Qa, axis, 1), self.shifted(Qa, axis, -1)
        for side, v in ((0, lo), (1, hi)):
            if self.q["bc"][2 * axis + side] == 2:
                dim = v.dim() - 1 - axis
                v.narrow(dim, 0 if side == 0 else v.shape[dim] - 1, 1).fill_(self.ghost_Q[axis])
        return torch.where(ua > 0, Qa - lo, hi - Qa)

    def collide(self):
        q, D = self.q, self.D
        rho, u, T = self.moments()
        dQ = [self.gradient(rho * u[a] * (1.0 - 3.0 * T - u[a] ** 2), u[a], a) for a in range(D)]
        P = rho * T
        mu = q["mu0"] * (T / q["T_scale"]) ** q["mu_exp"] if q["mu_exp"] else torch.full_like(T, q["mu0"])
        w = 2.0 * P / (2.0 * mu + P)
        w1 = 2.0 * q["Pr"] * w / (2.0 - w + q["Pr"] * w)
        X = self.factors(u, T)
        X_ex = self.factors(u, T, [(2.0 - w) / (2.0 * rho * w) * d for d in dQ])
        S = [_gpsi(u[a], T) for a in range(D)] + [[torch.zeros_like(T)] * 3] * (3 - D)
        # q* - q^eq = u . (P - P^eq + div Q~ / 2)
        dq = []
        for a in range(D):
            t = torch.zeros_like(T)
            for b in range(D):
                Pab = sum(c[a] * c[b] * self.f[i] for i, c in enumerate(self.c) if c[a] * c[b])
                t = t + u[b] * (Pab - rho * u[a] * u[b] - (P - 0.5 * dQ[a] if a == b else 0.0))
            dq.append(t)
        for i, c in enumerate(self.c):
            self.f[i] += w * (self.f_dir(c, rho, X_ex) - self.f[i])
            ge = self.g_dir(c, rho, T, X, S)
            self.g[i] += w1 * (ge - self.g[i])
            if sum(abs(x) for x in c) == 1:
                a = next(k for k in range(3) if c[k])
                self.g[i] -= 0.5 * (w - w1) * c[a] * dq[a]

    def step(self, n):
        for _ in range(n):
            self.stream()
            self.collide()

    def pairs(self, store, swapped=False):
        """The store's contents: Q planes of pairs (f, g), deviations from the rest state for the 16-bit stores."""
        f, g = self.f, self.g
        if store in ("f16dev", "bf16dev"):
            one = torch.ones((), device=DEV, dtype=F64)
            rf, rg = self.equilibrium(one, torch.zeros(self.D, device=DEV, dtype=F64), one * self.q["T_scale"])
            shape = (self.Q,) + (1,) * (f.dim() - 1)
            f, g = f - rf.reshape(shape), g - rg.reshape(shape)
        if swapped:   # the single store after an even number of steps: each pair in the opposite direction's plane
            f, g = f.flip(0), g.flip(0)
        return torch.stack([f, g], -1).reshape(-1)

    def statistics(self):
        rho, u, T = self.moments()
        N, D = rho.numel(), self.D
        G = [[0.5 * (torch.roll(u[a], -1, 2 - b) - torch.roll(u[a], 1, 2 - b)) for b in range(D)] for a in range(D)]
        uu = sum(x * x for x in u)
        w2 = (G[2][1] - G[1][2]) ** 2 + (G[0][2] - G[2][0]) ** 2 + (G[1][0] - G[0][1]) ** 2
        mu = self.q["mu0"] * (T / self.q["T_scale"]) ** self.q["mu_exp"]
        d = dict(rho_mean=rho.mean(), K=0.5 * (rho * uu).mean(), u_rms=torch.sqrt(uu.mean() / D), theta_rms=torch.sqrt(((G[0][0] + G[1][1] + G[2][2]) ** 2).mean()),
                 T_mean=T.mean(), dudx2=(G[0][0] ** 2).mean(), omega_rms=torch.sqrt(w2.mean()), enstrophy=0.5 * w2.mean(), dissipation=(mu * w2).mean(),
                 rho_rms=rho.std(correction=0), T_rms=T.std(correction=0))
        d["lambda"] = torch.sqrt((u[0] ** 2).sum() / (G[0][0] ** 2).sum())
        d["Re_lambda"] = d["rho_mean"] * d["u_rms"] * d["lambda"] / self.q["mu0"]
        totals = [rho.sum()] + [(rho * u[a]).sum() for a in range(D)] + [torch.zeros((), device=DEV, dtype=F64)] * (3 - D) + [self.g.sum()]
        return torch.stack(totals), torch.stack([d[k] for k in STATS])


def exact(case, seed):
    kind, store, n = case["kind"], case["store"], case.get("steps", 0)
    if kind == "ensemble":
        out = []
        for q in _members(case, seed):
            e = Exact(q)
            e.step(n)
            out.append(e.pairs(store))
        return torch.cat(out)
    e = Exact(_problem(case, seed))
    e.step(n)
    if kind in ("tube", "snapshot"):
        rho, u, T = e.moments()
        fields = [rho.reshape(-1), torch.stack(u).reshape(-1), T.reshape(-1)]
        if kind == "tube":
            return tuple(fields)
        totals, stats = e.statistics()
        return fields, totals, stats
    out = e.pairs(store, swapped=kind == "inplace")
    return (out, e.statistics()[1]) if kind == "history" else out
