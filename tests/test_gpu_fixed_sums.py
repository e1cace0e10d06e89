"""GPU test of the FP64 moments, which are summed as 64-bit integers on the scale of the node's largest
moving population: against exact sums, for populations of either sign, zero, far apart, of every
scale, and with values that are not finite.  Bounds: 27 terms off by 2^-57 of the largest each,
two roundings, and for u and T the quotient's."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("scale", [0, 300, -300, 990, -880, -1005])
@pytest.mark.parametrize("kind", ["near", "spread", "signs", "zeros"])
def test_fields_of_given_populations(D, scale, kind):
    import torch
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm as E
    nx, ny, nz = (7, 3, 1) if D == 2 else (5, 3, 2)
    Q, N = (9, nx * ny) if D == 2 else (27, nx * ny * nz)
    g = E.Solver.from_case(C.random_smooth(D, nx, ny, nz, seed=3, mu0=0.01, du=0.05, u0=(0.05, 0.0, 0.0)), store="f64")
    rng = np.random.default_rng(Q + abs(scale))
    pop = g.pop_a.view(torch.float64).cpu().numpy()[:2 * Q * N].reshape(Q, N, 2).copy()
    if kind == "spread":
        pop *= 2.0 ** rng.uniform(-60, 0, pop.shape)
    elif kind == "signs":
        pop[Q // 2] *= 40
        pop *= rng.choice([-1.0, 1.0], pop.shape) ** (np.arange(Q) != Q // 2)[:, None, None]
    elif kind == "zeros":
        pop[rng.random(pop.shape) < 0.5] = 0.0
        pop[Q // 2] += 0.1
        pop[: Q // 2, 0] = pop[Q // 2 + 1:, 0] = 0.0
    pop = np.ldexp(pop, scale)
    g.pop_a.view(torch.float64)[:2 * Q * N].copy_(torch.from_numpy(pop.ravel()))
    rho, u, T = (torch.empty(k * N, dtype=torch.float64, device="cuda") for k in (1, D, 1))
    g.fields_device(rho, u, T)
    rho, u, T = rho.cpu().numpy(), u.cpu().numpy().reshape(D, N), T.cpu().numpy()
    c = [[(i // 3 ** a) % 3 - 1 for a in range(D)] for i in range(Q)]
    for n in range(N):
        f, e = ([Fraction(float(v)) for v in pop[:, n, k]] for k in (0, 1))
        r, size, size_e = sum(f), sum(map(abs, f)), sum(map(abs, e))
        tiny = Fraction(2) ** -1074 * 30
        assert abs(Fraction(float(rho[n])) - r) <= EPS * size + tiny
        if abs(r) < EPS * 2 ** 10 * size or r == 0 or scale < -1000:
            continue
        w = float(size / abs(r))
        ue = [float(sum(ca[a] * v for ca, v in zip(c, f)) / r) for a in range(D)]
        for a in range(D):
            assert abs(u[a, n] - ue[a]) <= 4 * EPS * w * (1 + abs(ue[a]))
        en = float(sum(e) / r)
        bound = 8 * EPS * w * (float(size_e / abs(r)) + abs(en) + (1 + sum(abs(v) for v in ue)) ** 2)
        assert abs(T[n] - 0.4 * (en - 0.5 * sum(v * v for v in ue))) <= bound
    g.close()


@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_values_that_are_not_finite_stay_so(D, bad):
    import torch
    from paper_2102_09512_gb300 import elbm as E
    Q, nx = (9, 33) if D == 2 else (27, 33)
    c = C.random_smooth(D, nx, 2, 1 if D == 2 else 3, seed=3, mu0=0.01, du=0.05)
    N = nx * 2 * (1 if D == 2 else 3)
    for comp in (0, 1):
        g = E.Solver.from_case(c, store="f64")
        g.pop_a.view(torch.float64)[2 * ((Q - 1) * N + 40) + comp] = bad
        rho, u, T = (torch.empty(k * N, dtype=torch.float64, device="cuda") for k in (1, D, 1))
        with pytest.raises(Exception):
            g.fields_device(rho, u, T)
            g.sync()
        assert not bool(torch.isfinite(T[40])) and bool(torch.isfinite(T[39])) and bool(torch.isfinite(T[41]))
        g.close()
