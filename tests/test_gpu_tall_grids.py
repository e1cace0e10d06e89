"""GPU tests of grids with more tiles along one axis than the second and third dimension of a launch
hold (65535): what ran as one-dimensional launches takes them."""
import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm
    return elbm


@pytest.mark.parametrize("store", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(3, 600001), (40, 524289)])
def test_statistics_of_a_tall_sheet(E, store, nx, ny):
    """Against the same sums on the host; bound as in test_gpu_diagnostics.py."""
    c = C.random_smooth(2, nx, ny, 1, seed=64, mu0=0.01, du=0.05)
    g = E.Solver.from_case(c, store=store)
    g.set_kernel(E.ELBM_KERNEL_TWOPASS)
    g.step(2)
    dev = g.turbulence_stats()
    rho, u, T = g.fields()
    u, rho = u.reshape(2, ny, nx), rho.reshape(ny, nx)
    d = lambda a, ax: 0.5 * (np.roll(a, -1, ax) - np.roll(a, 1, ax))
    ref = dict(rho_mean=rho.mean(), T_mean=T.mean(), K=0.5 * (rho * (u ** 2).sum(0)).mean(), dudx2=(d(u[0], 1) ** 2).mean(),
               omega_rms=np.sqrt(((d(u[1], 1) - d(u[0], 0)) ** 2).mean()), theta_rms=np.sqrt(((d(u[0], 1) + d(u[1], 0)) ** 2).mean()))
    for k, v in ref.items():
        assert dev[k] == pytest.approx(v, rel=2.0 ** -40, abs=1e-18), k
    g.close()
