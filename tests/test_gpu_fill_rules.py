"""GPU tests of the marches that the allocation-free step and the single store choose by the share of
the tiles' threads that have nodes: against the two passes, on ragged grids on either side of the rules
(tiles whose last column or row is one node wide).  Bounds as in test_gpu_noalloc_schedules.py and
test_gpu_aa_march.py."""
import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

U0 = (0.09, -0.07, 0.06)


@pytest.fixture(scope="module")
def E():
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm
    return elbm


def close(got, ref, tol):
    for x, y in zip(got, ref):
        assert np.linalg.norm(np.ravel(x) - np.ravel(y)) <= tol * np.linalg.norm(np.ravel(y))


@pytest.mark.parametrize("store,tol", [("f32", 1e-6), ("f16dev", 1e-3), ("bf16dev", 8e-3)])
@pytest.mark.parametrize("shape", [(97, 25, 20), (62, 47, 9), (61, 45, 53), (40, 40, 40), (33, 600, 1), (80, 400, 1), (129, 601, 1)])
def test_allocation_free_step(E, shape, store, tol):
    import torch
    D = 3 if shape[2] > 1 else 2
    c = C.random_smooth(D, *shape, seed=93, mu0=0.01, mu_exp=0.76, du=0.05, u0=U0, bc=(1, 1, 0, 0, 0, 0))
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
    close(chk.fields(), ref.fields(), tol)
    ref.close()
    chk.close()


@pytest.mark.parametrize("store,tol", [("f32", 5e-6), ("f16dev", 1e-3), ("bf16dev", 8e-3)])
@pytest.mark.parametrize("shape", [(65, 65, 260), (97, 129, 90), (70, 65, 71), (60, 17, 900)])
def test_single_store(E, shape, store, tol):
    c = C.random_smooth(3, *shape, seed=152, mu0=0.01, du=0.05, u0=U0)
    aa = E.Solver.from_case(c, store=store, layout=E.ELBM_LAYOUT_AA)
    pp = E.Solver.from_case(c, store=store)
    pp.set_kernel(E.ELBM_KERNEL_TWOPASS)
    for n in (1, 2):
        aa.step(n)
        pp.step(n)
        close(aa.fields(), pp.fields(), tol)
    aa.close()
    pp.close()
