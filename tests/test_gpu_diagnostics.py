"""GPU tests of the diagnostics' arithmetic: the table-driven power functions of the
viscosity law and the FP64 reciprocal against extended precision, the totals against exactly rounded sums of the
stored populations, and the statistics at grids that are ragged against their tiles."""
import math
import os
import subprocess

import numpy as np
import pytest

from paper_2102_09512_gb300 import cases as C

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def E():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2102_09512_gb300 import build as B
    B.build()
    from paper_2102_09512_gb300 import elbm
    return elbm


POW_PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "elbm_node.cuh"
__global__ void run(const double* x, const double* e, double* y, double* h, double* l, double* q, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    y[i] = elbm::pow_pos(x[i], e[i]);
    q[i] = elbm::recip(e[i] * x[i]);
    const float eh = (float)e[i];
    elbm::Df r = {-1.f, 0.f};
    if (!elbm::pow_pos_df((float)x[i], {eh, (float)(e[i] - (double)eh)}, r)) r = {-1.f, 0.f};
    h[i] = r.h;
    l[i] = r.l;
}
int main(int argc, char** argv) {
    const int n = atoi(argv[1]);
    std::vector<double> b(2 * n), o(4 * n);
    if (fread(b.data(), 8, 2 * n, stdin) != (size_t)(2 * n)) return 2;
    double* d;
    if (cudaMalloc(&d, 6 * n * sizeof(double)) != cudaSuccess) return 3;
    cudaMemcpy(d, b.data(), 2 * n * sizeof(double), cudaMemcpyHostToDevice);
    run<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, d + 3 * n, d + 4 * n, d + 5 * n, n);
    if (cudaMemcpy(o.data(), d + 2 * n, 4 * n * sizeof(double), cudaMemcpyDeviceToHost) != cudaSuccess) return 4;
    return fwrite(o.data(), 8, 4 * n, stdout) == (size_t)(4 * n) ? 0 : 5;
}
"""


def test_power_functions(tmp_path):
    """pow_pos: half an ulp each from the table entry and the final addition and less than a
    half from everything carried in two doubles, so 1.5 ulp; the pair form: its logarithm
    times the exponent is good to 2^-45 of its size (at most 60, in use below 8), so 2^-41
    relative for |e log2 x| <= 8.  x includes both sides of every table boundary near 1.  recip:
    the iteration's last addition rounds once, its factors leave less than another half ulp."""
    from paper_2102_09512_gb300 import build as B
    src = tmp_path / "p.cu"
    src.write_text(POW_PROGRAM)
    exe = str(tmp_path / "p")
    subprocess.run([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "-I", B.CSRC, "-I", B.INCLUDE, "-o", exe, str(src)],
                   check=True)
    rng = np.random.default_rng(3)
    edges = np.concatenate([np.nextafter(1 + np.arange(129) / 128, s) for s in (0.0, 1.0, 4.0)])
    x = np.concatenate([edges, edges / 2, rng.uniform(0.3, 3.0, 100000), np.exp2(rng.uniform(-6, 6, 100000)), [1.0, 0.5, 2.0]])
    x = x.astype(np.float32).astype(np.float64)   # the same argument for both
    e = np.where(np.arange(x.size) % 2, 0.76, rng.uniform(-1.3, 1.3, x.size))
    e[-3:] = 0.76
    out = subprocess.run([exe, str(x.size)], input=np.concatenate([x, e]).tobytes(), stdout=subprocess.PIPE, check=True)
    y, h, l, q = np.frombuffer(out.stdout).reshape(4, -1)
    ref = np.power(x.astype(np.longdouble), e.astype(np.longdouble))
    assert float(np.max(np.abs(y - ref) / np.spacing(np.abs(y)))) <= 1.5
    r = 1.0 / (e * x)
    assert np.max(np.abs(q - r) / np.spacing(np.abs(r))) <= 1.0
    assert np.all(h > 0)
    assert float(np.max(np.abs(h.astype(np.longdouble) + l - ref) / ref)) <= 2.0 ** -41


@pytest.mark.parametrize("store", ["f64", "f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (45, 3, 1), (2048, 1, 1), (33, 9, 7), (2049, 3, 1), (61, 45, 53)])
def test_totals_equal_exact_sums(E, store, shape):
    """elbm_conservation against exactly rounded sums (math.fsum) of the stored populations, over
    pair counts around the run of a work unit (2048, FP64 4096) and below it.  The result is
    compensated to the last bit for the FP32-arithmetic stores, but for the rest state's sums,
    held in FP32; FP64 sums runs of 16 pairs plainly (error below 16 x 2^-53)."""
    D = 3 if shape[2] > 1 else 2
    c = C.random_smooth(D, *shape, seed=61, mu0=0.01)
    g = E.Solver.from_case(c, store=store)
    g.step(2)
    got = g.conservation()
    raw = g.get_populations()
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
        T, rho = g.params.T_ref, g.params.rho_ref
        ref[0] += N * rho
        ref[4] += N * rho * (T / (c.gamma - 1.0))
    tol = {"f64": 16 * 2.0 ** -53, "f32": 2.0 ** -52}.get(store, 27 * 2.0 ** -24)
    assert np.all(np.abs(got - ref) <= tol * ref[0]), (got, ref)
    g.close()


@pytest.mark.parametrize("store", ["f64", "f32"])
@pytest.mark.parametrize("shape,bc", [((33, 9, 7), (0,) * 6), ((32, 8, 33), (1, 1, 0, 0, 1, 1)), ((5, 70, 3), (0, 0, 1, 1, 0, 0)),
                                      ((65, 17, 1), (1, 1, 1, 1, 0, 0))])
def test_statistics_on_ragged_grids(E, store, shape, bc):
    """The device statistics against the same sums taken on the host in FP64 from the extracted
    fields (ghosts by the boundary map).  FP32 stores: the fields are the FP32 node values
    themselves, so only the terms' rounding is left (2^-40 covers it; the rms values of rho
    and T are differences of sums and keep fewer digits)."""
    D = 3 if shape[2] > 1 else 2
    c = C.random_smooth(D, *shape, seed=62, mu0=0.01, mu_exp=0.76, bc=bc)
    g = E.Solver.from_case(c, store=store)
    g.step(3)
    dev = g.turbulence_stats()
    rho, u, T = g.fields()
    sh = (c.nz, c.ny, c.nx)
    rho, T, u = rho.reshape(sh), T.reshape(sh), u.reshape((D,) + sh)

    def d(a, axis):
        per = bc[2 * (2 - axis)] == 0
        w = [(0, 0)] * 3
        w[axis] = (1, 1)
        p = np.pad(a, w, mode="wrap" if per else "edge")
        n = a.shape[axis]
        return 0.5 * (np.take(p, np.arange(2, n + 2), axis) - np.take(p, np.arange(n), axis))

    G = [[d(u[a], 2 - b) for b in range(D)] for a in range(D)]
    theta = sum(G[a][a] for a in range(D))
    w2 = (G[1][0] - G[0][1]) ** 2
    if D == 3:
        w2 = w2 + (G[2][1] - G[1][2]) ** 2 + (G[0][2] - G[2][0]) ** 2
    uu = (u ** 2).sum(0)
    mu = c.mu0 * (T / c.T0) ** c.mu_exp
    ref = dict(rho_mean=rho.mean(), K=0.5 * (rho * uu).mean(), u_rms=np.sqrt(uu.mean() / D), theta_rms=np.sqrt((theta ** 2).mean()),
               T_mean=T.mean(), dudx2=(G[0][0] ** 2).mean(), omega_rms=np.sqrt(w2.mean()), enstrophy=0.5 * w2.mean(),
               dissipation=(mu * w2).mean())
    for k, v in ref.items():
        assert dev[k] == pytest.approx(v, rel=2.0 ** -40, abs=1e-18), k
    assert dev["rho_rms"] == pytest.approx(rho.std(), rel=1e-9)
    assert dev["T_rms"] == pytest.approx(T.std(), rel=1e-9)
    g.close()
