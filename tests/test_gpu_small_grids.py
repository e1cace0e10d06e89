"""GPU tests of what the default schedule runs on small D2Q9 grids and of the rule that chooses
it: one strip of 30 nodes per CTA (FP64: its arithmetic shared by four warps), tiles, short row
segments and the FP64 two passes, at the sizes where a strip is full, one node short or one
node over, and in every option of the collision.  Bounds as in test_gpu_parity.py."""
import numpy as np
import pytest

import oracle as O
from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "f32": 1e-5, "f16dev": 1e-3, "bf16dev": 8e-3}
U0 = (0.09, -0.07, 0.0)


@pytest.fixture(scope="module")
def E():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2102_09512_gb300 import build as B
    B.build()
    O.build()
    from paper_2102_09512_gb300 import elbm
    return elbm


def rel_l2(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


def case(nx, ny, bc, cv=None, mu_exp=0.0):
    c = C.random_smooth(2, nx, ny, 1, seed=171 + nx, mu0=0.01, mu_exp=mu_exp, du=0.05, u0=U0, bc=bc)
    c.fixed = (1.0, U0[0], U0[1], 0.0, 0.15)
    c.cv = cv
    return c


def check(E, c, store, steps, deriv=0, kernel=0):
    s = O.init(O.Params(D=2, nx=c.nx, ny=c.ny, nz=1, gamma=c.gamma, Pr=c.Pr, mu0=c.mu0, T0=c.T0, mu_exp=c.mu_exp, bc=c.bc,
                        fixed=c.fixed, cv=c.cv, deriv=deriv), c.rho, c.u, c.T)
    O.step(s, steps)
    g = E.Solver.from_case(c, store=store, deriv=deriv)
    g.set_kernel(kernel)
    g.step(steps)
    for a, b in zip(g.fields(), O.fields(s)):
        assert rel_l2(a, b) <= TOL[store], (store, c.nx, c.ny, c.bc)
    if store in ("f64", "f32"):   # the 16-bit stores round the state after its totals were taken
        t, ref = g.step_totals(), g.conservation()
        assert np.allclose(t, ref, rtol=0, atol=(1e-13 if store == "f64" else 2e-6) * abs(ref[0]))
    g.close()


@pytest.mark.parametrize("store", list(TOL))
@pytest.mark.parametrize("bc", [(0,) * 6, (1, 1, 1, 1, 0, 0), (2, 1, 0, 0, 0, 0), (2, 1, 2, 1, 0, 0)])
@pytest.mark.parametrize("nx,ny", [(1, 5), (2, 1), (29, 4), (30, 3), (31, 2), (60, 5), (91, 1)])
def test_strips(E, nx, ny, bc, store):
    check(E, case(nx, ny, bc), store, 25)


@pytest.mark.parametrize("store", ["f64", "f32"])
@pytest.mark.parametrize("deriv,cv,mu_exp", [(1, None, 0.0), (0, (1.0, 4.0, -4.0, 5.0), 0.0), (0, None, 0.76)])
def test_strip_options(E, store, deriv, cv, mu_exp):
    check(E, case(47, 6, (1, 1, 0, 0, 0, 0), cv, mu_exp), store, 25, deriv)


@pytest.mark.parametrize("store", ["f64", "f32", "f16dev"])
@pytest.mark.parametrize("nx,ny", [(150, 200), (180, 203), (608, 256), (616, 257), (700, 333)])
@pytest.mark.parametrize("kernel", [0, 1])
def test_sizes_around_the_rule(E, nx, ny, store, kernel):
    """Strip and tile counts on either side of the rule's limits, and just above them, where
    the march runs segments of a few rows and FP64 its two passes."""
    check(E, case(nx, ny, (0,) * 6 if nx % 2 else (1, 1, 0, 0, 0, 0)), store, 6, kernel=kernel)


@pytest.mark.parametrize("store", ["f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("bc", [(0,) * 6, (1, 1, 1, 1, 0, 0), (2, 1, 2, 1, 0, 0)])
@pytest.mark.parametrize("nx,ny,tz", [(257, 40, 7), (512, 33, 16), (255, 9, 1), (6, 30, 10), (1, 12, 5), (770, 21, None)])
def test_row_march(E, nx, ny, tz, bc, store):
    """The row march (two nodes a thread for the 16-bit stores) forced on strips that end on a
    pair, between the nodes of one and one node over, with rows on and off 8-byte boundaries and
    fixed faces, and segments of one row."""
    c = case(nx, ny, bc)
    s = O.init(O.Params(D=2, nx=nx, ny=ny, nz=1, gamma=c.gamma, Pr=c.Pr, mu0=c.mu0, T0=c.T0, mu_exp=0.0, bc=bc,
                        fixed=c.fixed), c.rho, c.u, c.T)
    O.step(s, 20)
    g = E.Solver.from_case(c, store=store)
    g.set_tile_z(ny if tz is None else tz)
    g.step(20)
    for a, b in zip(g.fields(), O.fields(s)):
        assert rel_l2(a, b) <= TOL[store], (store, nx, ny, bc)
    g.close()


@pytest.mark.parametrize("store", ["f64", "f32"])
def test_one_grid_s_share_of_an_sm_beside_another_s(E, store):
    """The shared memory that spreads a grid's CTAs goes with the grid's size: grids of 1, 2 and 8
    CTAs to an SM, one more than that, FP64 two passes on either side of their limits, stepped
    in turn and from graphs captured before the others ran, match each alone."""
    sizes = [(30, 152), (30, 153), (60, 152), (29, 1216), (152, 128), (153, 128), (190, 205), (389, 400)]
    cases = [case(nx, ny, (1, 1, 0, 0, 0, 0)) for nx, ny in sizes]
    alone = []
    for c in cases:
        g = E.Solver.from_case(c, store=store)
        g.step(8)
        alone.append(g.pop_a.clone())
        g.close()
    gs = [E.Solver.from_case(c, store=store) for c in cases]
    for g in gs[::2]:
        g.set_step_graph(2)
    for _ in range(4):
        for g in gs:
            g.step(2)
    for g, a in zip(gs, alone):
        assert bool((g.pop_a == a).all())
        g.close()
