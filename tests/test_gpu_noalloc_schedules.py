"""GPU test of the allocation-free step above the size from which it runs the default schedule of
a handle: two steps against the two-pass handle, in every lattice and store, on grids whose fused
kernels have more CTAs than the two-pass ones (rows of one tile, short segments)."""
import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

# two steps of FP64/FP32 rounding; a storage rounding that falls the other way is one unit of the
# 16-bit deviation (2^-11, 2^-8), about the size of these fields' deviations from rest
TOL = {"f64": 1e-14, "f32": 1e-6, "f16dev": 1e-3, "bf16dev": 8e-3}


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


@pytest.mark.parametrize("store", list(TOL))
@pytest.mark.parametrize("shape,bc", [((32, 32, 16), (0,) * 6), ((33, 9, 60), (1, 1, 0, 0, 1, 1)), ((1, 40, 420), (0,) * 6),
                                      ((128, 128, 1), (0,) * 6), ((20000, 1, 1), (2, 1, 0, 0, 0, 0)),
                                      ((700, 400, 1), (1, 1, 1, 1, 0, 0))])
def test_noalloc_above_the_small_grids(E, shape, bc, store):
    import torch
    D = 3 if shape[2] > 1 else 2
    c = C.random_smooth(D, *shape, seed=92, mu0=0.01, mu_exp=0.76, du=0.05, u0=(0.09, -0.07, 0.06), bc=bc)
    c.fixed = (1.0, 0.09, -0.07, 0.0, 0.15)
    ref = E.Solver.from_case(c, store=store)
    ref.set_kernel(E.ELBM_KERNEL_TWOPASS)
    start = ref.get_populations()
    ref.step(2)
    a = torch.from_numpy(start).cuda()
    b = torch.empty_like(a)
    stream = torch.cuda.current_stream().cuda_stream
    for src, dst in ((a, b), (b, a)):
        assert E.elbm_step_noalloc(ref.params, src.data_ptr(), dst.data_ptr(), stream) == E.ELBM_OK
    torch.cuda.synchronize()
    chk = E.Solver(ref.params)
    chk.set_populations(a.cpu().numpy())
    for x, y in zip(chk.fields(), ref.fields()):
        assert rel_l2(x, y) <= TOL[store]
    ref.close()
    chk.close()
