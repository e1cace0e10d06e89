"""GPU test of the 16-bit stores' bits: populations after some steps against recorded digests of the
kernels that march one node a thread.  A last bit of FP32 arithmetic is now and then a last bit of
the store, so a kernel whose operations round otherwise moves some of these values.  The fields are whole
numbers over powers of two, so that no library function takes part in them."""
import hashlib

import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu


def fields(D, nx, ny, nz, bc=(0,) * 6, mu_exp=0.0, uy=-0.0625):
    z, y, x = (a.astype(np.int64) for a in np.indices((nz, ny, nx)))

    def wave(k, n, amp):   # a triangular wave along every axis and an uneven remainder
        t = sum(np.abs((a * k + 7 * k * (i + 1)) % 64 - 32) for i, a in enumerate((x, y, z)))
        return amp * (t / 128.0 + ((x * 37 + y * 91 + z * 53 + n) % 32) / 4096.0 - 0.25)

    rho, T = 1.0 + wave(1, 3, 0.0625), 0.15625 * (1.0 + wave(2, 5, 0.03125))
    u = np.stack([c + wave(1 + a, 11 * a, 0.0625) for a, c in enumerate((0.09375, uy, 0.03125)[:D])])
    return C.Case("bits", D, nx, ny, nz, rho, u, T, Pr=0.75, mu0=0.015625, T0=0.15625, mu_exp=mu_exp, bc=bc,
                  fixed=(1.0, 0.09375, -0.0625, 0.0, 0.15625))


ZERO, FIXED = (1, 1, 0, 0, 0, 0), (2, 1, 1, 1, 0, 0)
CASES = {
    "march": (2, 1280, 1021, 1, {}),
    "march odd": (2, 1023, 1280, 1, dict(bc=ZERO, uy=0.0625)),
    "march power": (2, 1536, 1024, 1, dict(mu_exp=0.75)),
    "march fixed": (2, 1281, 1024, 1, dict(bc=FIXED)),
    "box": (3, 64, 48, 50, {}),
    "box ragged": (3, 61, 45, 53, dict(bc=(0, 0, 1, 1, 0, 0))),
    "box power": (3, 128, 128, 128, dict(mu_exp=0.75)),
}
DIGESTS = {
    ("march", "f16dev"): "6e730a1ed1c8131f",
    ("march odd", "f16dev"): "96070cd4fece85c7",
    ("march power", "f16dev"): "4660317675a5de20",
    ("march fixed", "f16dev"): "2853793470481118",
    ("box", "f16dev"): "f3e01ed74844c1a6",
    ("box ragged", "f16dev"): "121fee3614abb9a0",
    ("box power", "f16dev"): "2aedfc4eb5a3e4b1",
    ("ensemble", "f16dev"): "1fe2526b5b39e172",
    ("ensemble fixed", "f16dev"): "1c870966f26a7bae",
    ("march", "bf16dev"): "0975a9f7f283ba13",
    ("march odd", "bf16dev"): "01f7224a9352b612",
    ("march power", "bf16dev"): "1b31b0bc5821b08f",
    ("march fixed", "bf16dev"): "9dd63d161c44793a",
    ("box", "bf16dev"): "9f39702a9b2c58e9",
    ("box ragged", "bf16dev"): "eadd8cf2a6eb4bf7",
    ("box power", "bf16dev"): "3f79b5c82e69d0bf",
    ("ensemble", "bf16dev"): "6d1f8619362bd617",
    ("ensemble fixed", "bf16dev"): "663ca5a5385dcb04",
}


def digest(E, name, store, steps=6):
    D, nx, ny, nz, kw = CASES[name]
    g = E.Solver.from_case(fields(D, nx, ny, nz, **kw), store=store, rho_ref=1.0, T_ref=0.15625)
    g.set_tile_z(16)
    c = fields(D, nx, ny, nz, **kw)
    g.set_fields(c.rho, c.u, c.T)
    g.step(steps)
    out = hashlib.sha256(np.ascontiguousarray(g.get_populations()).tobytes()).hexdigest()[:16]
    g.close()
    return out


def ensemble_digest(E, store, fixed, steps=6):
    cs = [fields(2, 300, 257, 1), fields(2, 311, 200, 1, bc=FIXED if fixed else ZERO), fields(2, 128, 96, 1)]
    e = E.Ensemble.from_cases(cs, store=store)
    e.set_schedule(32, 2)
    e.step(steps)
    e.sync()
    return hashlib.sha256(np.ascontiguousarray(e.pop_a.cpu().numpy()).tobytes()).hexdigest()[:16]


@pytest.fixture(scope="module")
def E():
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm
    return elbm


@pytest.mark.parametrize("store", ["f16dev", "bf16dev"])
@pytest.mark.parametrize("name", list(CASES))
def test_populations_keep_their_bits(E, name, store):
    assert digest(E, name, store) == DIGESTS[name, store]


@pytest.mark.parametrize("store", ["f16dev", "bf16dev"])
@pytest.mark.parametrize("fixed", [False, True])
def test_ensembles_keep_their_bits(E, store, fixed):
    assert ensemble_digest(E, store, fixed) == DIGESTS["ensemble fixed" if fixed else "ensemble", store]
