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


def host_stats(c, D, rho, u, T):
    """The statistics' means in extended precision from node values on a periodic grid."""
    sh = (c.nz, c.ny, c.nx)
    rho, T, u = rho.astype(LD).reshape(sh), T.astype(LD).reshape(sh), u.astype(LD).reshape((D,) + sh)
    G = [[(np.roll(u[a], -1, 2 - b) - np.roll(u[a], 1, 2 - b)) / 2 for b in range(D)] for a in range(D)]
    theta = sum(G[a][a] for a in range(D))
    w2 = (G[1][0] - G[0][1]) ** 2
    if D == 3:
        w2 = w2 + (G[2][1] - G[1][2]) ** 2 + (G[0][2] - G[2][0]) ** 2
    uu = (u ** 2).sum(0)
    mu = LD(c.mu0) * (T / LD(c.T0)) ** LD(c.mu_exp)
    return dict(K=0.5 * (rho * uu).mean(), u_rms=np.sqrt(uu.mean() / D), theta_rms=np.sqrt((theta ** 2).mean()),
                dudx2=(G[0][0] ** 2).mean(), omega_rms=np.sqrt(w2.mean()), enstrophy=0.5 * w2.mean(),
                dissipation=(mu * w2).mean())


# Exponents whose T^mu_exp (T = 0.15) is below, and above, what FP32 holds, and whose lower bits are, and whose
# (T/T0)^mu_exp is (T0 = 15); deviations from rest so small that the squares of the velocities, or of
# their differences alone, are; and one state that floats hold.
# Bound 2^-46: the law takes T/T0, off by 2^-53, to the 60th power (2^-47); the sums are FP64.
@pytest.mark.parametrize("D,shape", [(3, (33, 9, 7)), (2, (65, 17, 1))])
@pytest.mark.parametrize("store,scale,mu_exp,T0", [("f32", 0, 60.0, 0.15), ("f32", 0, -60.0, 0.15), ("f32", 0, 40.0, 0.15),
                                                   ("f32", 0, 60.0, 15.0), ("f32", 0, 0.76, 0.15),
                                                   ("bf16dev", 2.0 ** -60, 0.76, 0.15), ("bf16dev", 2.0 ** -80, 0.76, 0.15),
                                                   ("bf16dev", 2.0 ** -40, 0.0, 0.15)])
def test_terms_outside_the_range_of_floats(E, store, scale, mu_exp, T0, D, shape):
    c = C.random_smooth(D, *shape, seed=9, mu0=0.01, du=0.05, u0=(0.09, -0.07, 0.06)[:D] + (0.0,) * (3 - D), mu_exp=mu_exp)
    c.T0 = T0
    g = E.Solver.from_case(c, store=store)
    if scale:   # populations rest + scale x (what the case has), exact: multiplied by a power of two
        raw = g.get_populations().view(np.uint16)
        v = (raw.astype(np.uint32) << 16).view(np.float32) * np.float32(scale)
        g.set_populations((v.view(np.uint32) >> 16).astype(np.uint16).view(np.uint8))
    dev = g.turbulence_stats()
    ref = host_stats(c, D, *g.fields())
    g.close()
    for k, v in ref.items():
        assert v > 0
        assert abs(LD(dev[k]) / v - 1) <= 2.0 ** -46, k


@pytest.mark.parametrize("store", ["f32", "f16dev"])
def test_dissipation_has_no_bias(E, store):
    """A state's dissipation is rounded some six times at the end (the factor of the law, mu0, the sums, the
    division), 2^-53 each to either side, so that the mean error of eight states is below 2^-52 unless the
    terms have one in common."""
    err = []
    for seed in range(8):
        c = C.random_smooth(3, 40, 41, 42, seed=seed, T0=0.13 + 0.01 * seed, mu0=0.01 + 0.003 * seed, du=0.05,
                            u0=(0.09, -0.07, 0.06), mu_exp=0.76)
        g = E.Solver.from_case(c, store=store)
        dev = g.turbulence_stats()
        err.append(float(LD(dev["dissipation"]) / host_stats(c, 3, *g.fields())["dissipation"] - 1))
        g.close()
    assert abs(np.mean(err)) <= 2.0 ** -52, err


def test_zeros_are_sums_of_zeros(E):
    """A flow that does not depend on x has no dilatation and no d u_x / d x, one at rest no velocity: their sums
    are exactly zero, and known to be from the one pass over the store (two launches, as for any state)."""
    for D, shape, u0 in ((3, (33, 9, 7), 0.05), (2, (65, 17, 1), 0.05), (2, (40, 8, 1), 0.0)):
        c = C.random_smooth(D, *shape, seed=9, mu0=0.01, mu_exp=0.76)
        c.rho[:], c.T[:], c.u[:] = 1.0, 0.15, 0.0
        c.u[0] = u0 * np.sin(2 * np.pi * np.arange(c.ny) / c.ny)[None, :, None]
        g = E.Solver.from_case(c, store="f32")
        before = g.launches
        s = g.turbulence_stats()
        assert g.launches - before == 2
        assert s["theta_rms"] == s["dudx2"] == 0.0 and (s["omega_rms"] > 0) == (s["dissipation"] > 0) == (s["K"] > 0) == (u0 > 0)
        g.close()
