"""GPU test of elbm_conservation against exactly rounded sums, at pair counts on either side of a
work unit (4096 pairs: its unchecked reads meet the checked ones of the last unit).

FP64 bound: a value is rounded to 2^-57 of the largest of its run of 16, to either side, and nothing else
but the result is: 8 standard deviations of N values of every direction that the sum takes, and the
result's rounding.  The FP32-arithmetic stores: as in test_gpu_diagnostics.py."""
import math

import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", ["f64", "f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("shape", [(4095, 1, 1), (64, 64, 1), (4097, 1, 1), (15, 13, 21), (16, 16, 16), (17, 241, 1), (32, 16, 16)])
def test_totals_around_a_work_unit(shape, store):
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm as E
    D = 3 if shape[2] > 1 else 2
    c = C.random_smooth(D, *shape, seed=67, mu0=0.01)
    g = E.Solver.from_case(c, store=store)
    g.step(2)
    got = g.conservation()
    raw = g.get_populations()
    g.close()
    N, Q = c.N, 27 if D == 3 else 9
    if store == "bf16dev":
        v = (raw.view(np.uint16).astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    else:
        v = raw.view({"f64": np.float64, "f32": np.float32, "f16dev": np.float16}[store]).astype(np.float64)
    v = v.reshape(Q, N, 2)
    vel = np.array([E.elbm_velocity(g.params.lattice, i) for i in range(Q)], dtype=np.float64)
    ref = [math.fsum(v[:, :, 0].ravel())] + [math.fsum((vel[:, a, None] * v[:, :, 0]).ravel()) for a in range(3)]
    ref.append(math.fsum(v[:, :, 1].ravel()))
    if store.endswith("dev"):
        ref[0] += N * g.params.rho_ref
        ref[4] += N * g.params.rho_ref * (g.params.T_ref / (c.gamma - 1.0))
    big = np.abs(v).max(axis=1)   # of every direction, f and g
    for k in range(5):
        if store == "f64":
            part = big[:, 1] if k == 4 else big[:, 0] * (1.0 if k == 0 else np.abs(vel[:, k - 1]))
            tol = 8 * 2.0 ** -57 * math.sqrt(N * float((part ** 2).sum())) + 2.0 ** -53 * abs(ref[k])
        else:
            tol = (2.0 ** -52 if store == "f32" else 27 * 2.0 ** -24) * ref[0]
        assert abs(got[k] - ref[k]) <= tol, (k, got[k], ref[k], tol)
