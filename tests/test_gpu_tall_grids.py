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


TOL = {"f64": 1e-14, "f32": 1e-6, "f16dev": 1e-3, "bf16dev": 8e-3}   # as in test_gpu_noalloc_schedules.py


@pytest.mark.parametrize("store", list(TOL))
@pytest.mark.parametrize("shape", [(1, 600000, 1), (1, 1, 600000), (1, 524281, 1)])
def test_allocation_free_step(E, store, shape):
    import torch
    c = C.random_smooth(3, *shape, seed=65, mu0=0.01, du=0.05)
    ref = E.Solver.from_case(c, store=store)
    ref.set_kernel(E.ELBM_KERNEL_TWOPASS)
    a = torch.from_numpy(ref.get_populations()).cuda()
    b = torch.empty_like(a)
    ref.step(2)
    for src, dst in ((a, b), (b, a)):
        assert E.elbm_step_noalloc(ref.params, src.data_ptr(), dst.data_ptr(), torch.cuda.current_stream().cuda_stream) == E.ELBM_OK
    torch.cuda.synchronize()
    chk = E.Solver(ref.params)
    chk.set_populations(a.cpu().numpy())
    for x, y in zip(chk.fields(), ref.fields()):
        assert np.linalg.norm(np.ravel(x) - np.ravel(y)) <= TOL[store] * np.linalg.norm(np.ravel(y))
    ref.close()
    chk.close()


@pytest.mark.parametrize("store", ["f32", "f16dev"])
@pytest.mark.parametrize("shape", [(1, 600000, 1), (2, 524281, 1)])
def test_single_store(E, store, shape):
    c = C.random_smooth(3, *shape, seed=66, mu0=0.01, du=0.05)
    aa = E.Solver.from_case(c, store=store, layout=E.ELBM_LAYOUT_AA)
    pp = E.Solver.from_case(c, store=store)
    pp.set_kernel(E.ELBM_KERNEL_TWOPASS)
    pp.set_fields(c.rho, c.u, c.T)
    aa.step(2)
    pp.step(2)
    for x, y in zip(aa.fields(), pp.fields()):
        assert np.linalg.norm(np.ravel(x) - np.ravel(y)) <= 5 * TOL[store] * np.linalg.norm(np.ravel(y))
    aa.close()
    pp.close()
