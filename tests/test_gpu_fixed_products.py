"""GPU tests of the FP64 collision whose products are formed in integers (the two passes on more
than one CTA to an SM), bounds as in test_gpu_parity.py: against the oracle, with populations of either
sign, and on other scales, where density and viscosity times a power of two give the same velocities."""
import numpy as np
import pytest

import oracle as O
from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

SIZES = {2: (181, 131, 1), 3: (31, 29, 27)}


def rel_l2(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


def run(c, steps):
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm as E
    g = E.Solver.from_case(c, store="f64")
    g.set_kernel(1)
    g.step(steps)
    out = g.fields()
    g.close()
    return out


@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("scale", [0, 150, 400, -150, -400])
@pytest.mark.parametrize("flow", [0.09, 0.5])
@pytest.mark.parametrize("mu_exp", [0.0, 0.76])
def test_steps(D, scale, flow, mu_exp):
    O.build()
    nx, ny, nz = SIZES[D]
    bc = (2, 1, 0, 0, 0, 0) if D == 2 else (0,) * 6
    c = C.random_smooth(D, nx, ny, nz, seed=5, mu0=0.01, mu_exp=mu_exp, du=0.03, u0=(flow, -0.07, 0.06 if D == 3 else 0.0), bc=bc)
    c.fixed = (1.0, flow, -0.07, 0.0, 0.15)
    s = O.init(O.Params(D=D, nx=nx, ny=ny, nz=nz, gamma=c.gamma, Pr=c.Pr, mu0=c.mu0, T0=c.T0, mu_exp=c.mu_exp, bc=c.bc,
                        fixed=c.fixed, cv=c.cv), c.rho, c.u, c.T)
    O.step(s, 10)
    f = 2.0 ** scale
    c.rho, c.mu0, c.fixed = c.rho * f, c.mu0 * f, (f, *c.fixed[1:])
    rho, u, T = run(c, 10)
    for a, b in zip((rho / f, u, T), O.fields(s)):
        assert rel_l2(a, b) <= 1e-12


@pytest.mark.parametrize("D", [2, 3])
def test_a_gas_at_rest_stays_at_rest(D):
    nx, ny, nz = SIZES[D]
    c = C.random_smooth(D, nx, ny, nz, seed=5, mu0=0.01, drho=0.0, du=0.0, dT=0.0)
    rho, u, T = run(c, 12)
    assert not np.any(u)
