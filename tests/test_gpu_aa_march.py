"""GPU tests of the in-place march of the AA layout (D3Q27 stores larger than the L2 cache, FP32
arithmetic): against the ping-pong two-pass schedule on grids ragged against its tiles and segments,
with tiles of one row or column and segments of one plane, with and without a tensor map, and
that a run repeats bit for bit (no thread reads a slot that another writes).  Bounds as in
test_gpu_aa.py; few steps, so that 16-bit roundings that differ have not grown."""
import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

SAME = {"f32": 5e-6, "f16dev": 1e-3, "bf16dev": 8e-3}
U0 = (0.09, -0.07, 0.06)


@pytest.fixture(scope="module")
def E():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm
    return elbm


def rel_l2(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


# every one above 64 MB of store (216 bytes a node in FP32, 108 in 16 bits)
@pytest.mark.parametrize("shape,store,tz", [((70, 65, 71), "f32", None), ((33, 300, 35), "f32", 8), ((400, 5, 160), "f32", 64),
                                            ((96, 64, 60), "f32", 1), ((32, 8, 1200), "f32", 128), ((256, 240, 6), "f32", 2),
                                            ((301, 257, 8), "f16dev", 3), ((128, 96, 50), "f16dev", 7),
                                            ((91, 81, 83), "bf16dev", None)])
@pytest.mark.parametrize("options", [{}, {"mu_exp": 0.76, "deriv": 1}, {"cv": (1.0, 4.0, -4.0, 5.0)}])
def test_march_equals_pingpong(E, shape, store, tz, options):
    c = C.random_smooth(3, *shape, seed=151, mu0=0.01, mu_exp=options.get("mu_exp", 0.0), du=0.05, u0=U0)
    c.cv = options.get("cv")
    deriv = options.get("deriv", 0)
    aa = E.Solver.from_case(c, store=store, layout=E.ELBM_LAYOUT_AA, deriv=deriv)
    if tz is not None:
        aa.set_tile_z(tz)
        aa.set_fields(c.rho, c.u, c.T)   # the initial collision marches the same segments
    pp = E.Solver.from_case(c, store=store, deriv=deriv)
    pp.set_kernel(E.ELBM_KERNEL_TWOPASS)
    for n in (1, 1, 2):
        aa.step(n)
        pp.step(n)
        for x, y in zip(aa.fields(), pp.fields()):
            assert rel_l2(x, y) <= SAME[store]
        assert rel_l2(aa.step_totals(), pp.step_totals()) <= SAME[store]
    state = aa.get_populations()
    aa.set_fields(c.rho, c.u, c.T)
    aa.step(4)
    assert np.array_equal(aa.get_populations(), state)
    aa.sync()
    aa.close()
    pp.close()
