"""GPU tests of the turbulence statistics of the FP32-arithmetic stores: the energy to the last bits of
FP64, and states whose terms leave the range of FP32."""
import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module")
def E():
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm
    return elbm


@pytest.mark.parametrize("store", ["f32", "bf16dev"])
@pytest.mark.parametrize("seed", [5, 6])
def test_energy_sums_have_no_bias(E, store, seed):
    """Against extended precision on the node values (fields): the sums are exact but for the rounding
    of the result, of the division by N and of the root (1.5 ulp each at most, 2^-53 x 3)."""
    c = C.random_smooth(3, 64, 64, 64, seed=seed, mu0=0.01, du=0.05, u0=(0.09, -0.07, 0.06))
    g = E.Solver.from_case(c, store=store)
    dev = g.turbulence_stats()
    rho, u, T = (a.astype(LD) for a in g.fields())
    g.close()
    uu = (u.reshape(3, -1) ** 2).sum(0)
    K, u_rms = 0.5 * (rho.ravel() * uu).sum() / uu.size, np.sqrt(uu.sum() / uu.size / 3)
    assert abs(dev["K"] / K - 1) <= 3 * 2.0 ** -53
    assert abs(dev["u_rms"] / u_rms - 1) <= 3 * 2.0 ** -53
