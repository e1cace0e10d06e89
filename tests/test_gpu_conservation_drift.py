"""GPU test of the FP64 step's mass and momentum over many steps: the integer sums and products of the
moments and the collision have no rounding with a sign.  N nodes whose sums are off by some 2^-53 to
either side in each of S steps move the mass of the grid by about 2^-53 sqrt(S / N) of itself, at most
5e-16 here; eight times that is allowed.  A rounding with a sign of 2^-60 a node and step
moves it by S 2^-60 = 9e-15."""
import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

S = 10000


# strips and tiles (integer sums), and the two passes on more CTAs than SMs (integer products too)
@pytest.mark.parametrize("shape,kernel", [((24, 24, 1), 0), ((24, 24, 1), 1), ((160, 131, 1), 1), ((28, 28, 28), 1), ((9, 8, 10), 2)])
def test_mass_does_not_drift(shape, kernel):
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm as E
    D = 3 if shape[2] > 1 else 2
    g = E.Solver.from_case(C.random_smooth(D, *shape, seed=8, mu0=0.02, du=0.05, u0=(0.09, -0.07, 0.06)), store="f64")
    g.set_kernel(kernel)
    before = g.conservation()
    g.step(S)
    after = g.conservation()
    g.close()
    N = np.prod(shape)
    tol = 8 * 2.0 ** -53 * max(1.0, (S / N) ** 0.5)
    for k in range(1 + D if N > S else 1):   # the momentum of the small grids is not that steady
        assert abs(after[k] - before[k]) <= tol * before[0], (k, (after[k] - before[k]) / before[0])
