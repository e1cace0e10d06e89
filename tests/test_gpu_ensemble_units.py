"""GPU test of the work units of the ensemble's row march: lattices of one row or column, of a strip
and one node more, of very uneven heights, fewer and more of them than CTAs run at once.  Bounds
as in test_gpu_parity.py."""
import numpy as np
import pytest

import oracle as O
from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5, "f16dev": 1e-3, "bf16dev": 8e-3}
U0 = (0.09, -0.07, 0.0)
MIXED = [(1, 7), (129, 2), (128, 257), (40, 700), (300, 31), (257, 1), (5, 64), (64, 1)]


def lattice(nx, ny, k):
    bc = [(0,) * 6, (1, 1, 0, 0, 0, 0), (0, 0, 1, 1, 0, 0)][k % 3]
    c = C.random_smooth(2, nx, ny, 1, seed=31 + k, mu0=0.01, du=0.05, u0=U0, bc=bc)
    c.fixed = (1.0, U0[0], U0[1], 0.0, 0.15)
    return c


@pytest.mark.parametrize("store", list(TOL))
@pytest.mark.parametrize("tile_y,ctas", [(32, 1), (64, 6), (128, 3)])
@pytest.mark.parametrize("sizes", [MIXED[3:4], MIXED, [(9, 5 + k % 3) for k in range(1000)] + MIXED])
def test_units_cover_every_lattice(sizes, tile_y, ctas, store):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2102_09512_gb300 import build as B
    B.build()
    O.build()
    from paper_2102_09512_gb300 import elbm as E
    cs = [lattice(nx, ny, k) for k, (nx, ny) in enumerate(sizes)]
    ens = E.Ensemble.from_cases(cs, store=store)
    ens.set_schedule(tile_y, ctas)
    ens.step(9)
    for k in sorted({0, 1 % len(cs), 500 % len(cs), *range(max(0, len(cs) - 8), len(cs))}):
        c = cs[k]
        s = O.init(O.Params(D=2, nx=c.nx, ny=c.ny, nz=1, gamma=c.gamma, Pr=c.Pr, mu0=c.mu0, T0=c.T0, mu_exp=c.mu_exp,
                            bc=c.bc, fixed=c.fixed, cv=c.cv), c.rho, c.u, c.T)
        O.step(s, 9)
        for a, b in zip(ens.fields(k), O.fields(s)):
            assert np.linalg.norm(np.ravel(a) - np.ravel(b)) <= TOL[store] * np.linalg.norm(np.ravel(b)), (k, c.nx, c.ny)
    ens.close()
