"""CPU checks of the segment planner (choose_segment in csrc/elbm_internal.h), which the
allocation-free step runs on every call: the lengths against the rule evaluated for every number of
segments, and the time a call takes on long grids; and of the rules that choose between a march and the
two passes (march_launches, aa_march_pays, noalloc_march_pays)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2102_09512_gb300", "csrc")

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include "elbm_internal.h"
using namespace elbm;
// best of all numbers of equal segments; ties keep the longer segment
static int every(double tiles, int n, int sms, int per, int fallback, int shortest) {
    const double slots = (double)sms * per;
    int best = fallback < n ? fallback : n;
    double top = -1.0;
    for (int nseg = 1; nseg <= n; ++nseg) {
        const int tz = (n + nseg - 1) / nseg;
        if (tz > 128) continue;
        if (tz < (n < shortest ? n : shortest)) break;
        const double waves = tiles * ((n + tz - 1) / tz) / slots;
        const double score = waves / std::ceil(waves) * tz / (tz + 2.0);
        if (score > top + 1e-9) { top = score; best = tz; }
    }
    return best;
}
int main() {
    long long bad = 0, seen = 0;
    const int per[] = {1, 2, 4, 6, 7}, shortest[] = {1, 16, 1000};
    for (int n = 1; n <= 5000; n += 1 + n / 40)
        for (int t = 1; t <= 70000; t += 1 + t / 6)
            for (int p : per)
                for (int s : shortest) {
                    ++seen;
                    bad += choose_segment(t, n, 152, p, 32, s) != every(t, n, 152, p, 32, s);
                }
    std::printf("%lld %lld\n", seen, bad);
    double worst = 1e9;   // the fastest of some repeats, us a call
    for (int r = 0; r < 20; ++r) {
        const auto a = std::chrono::steady_clock::now();
        int sum = 0;
        for (int k = 0; k < 50; ++k) sum += choose_segment(1 + k % 2, 65536 + k, 152, 7, 32) + choose_segment(8, 1000000 + k, 152, 4, 32);
        const double us = std::chrono::duration<double, std::micro>(std::chrono::steady_clock::now() - a).count() / 100 + (sum == 0);
        if (us < worst) worst = us;
    }
    std::printf("%f\n", worst);
    return 0;
}
"""


@pytest.fixture(scope="module")
def planned(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "p.cu", str(d / "p")
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", exe], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()


def test_lengths_are_the_best_of_all_segment_counts(planned):
    assert int(planned[0]) > 100000 and int(planned[1]) == 0


def test_planning_a_long_grid_takes_microseconds(planned):
    """At most 128 lengths are looked at, some ten nanoseconds each: below 20 us with a wide margin
    (a loop over the segment counts takes 400 us and more here)."""
    assert float(planned[2]) < 20.0


RULES = r"""
#include <cstdio>
#include <cstdlib>
#include "elbm_internal.h"
int main(int argc, char** argv) {
    elbm::KParams k{};
    const int D = atoi(argv[1]);
    k.nx = atoi(argv[2]); k.ny = atoi(argv[3]); k.nz = atoi(argv[4]); k.tz = atoi(argv[5]);
    if (D == -9) {   // CTAs of `stat` bytes that an SM holds with the share for k.nx CTAs on k.ny SMs (228 KB, 1 KB of it a CTA's)
        const size_t share = elbm::spread_share(k.nx, k.ny, k.nz);
        std::printf("%d\n", share ? (int)((228 * 1024) / (share + k.nz + 1024)) : 0);
        return 0;
    }
    if (D < 0) {   // plan_d2q9: store width of the strips, 64 bits, fixed faces
        k.N = (long long)k.nx * k.ny; k.tz = 32; k.has_fixed = atoi(argv[6]);
        elbm::plan_d2q9(k, 152, 4, 256, atoi(argv[5]));
        std::printf("%d\n", k.sched);
        return 0;
    }
    const double bytes = 27.0 * 8 * k.nx * k.ny * k.nz;
    std::printf("%d %d %d %d\n", elbm::march_launches(k, D, 8), elbm::aa_march_pays(k, 8, bytes),
                elbm::noalloc_march_pays(k, D, 128, 8), elbm::noalloc_march_pays(k, D, 256, 8));
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("rule")
    src, exe = d / "r.cu", str(d / "r")
    src.write_text(RULES)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src), "-o", exe], check=True)
    return lambda *a: [v == "1" if a[0] > 0 else int(v) for v in subprocess.run([exe, *map(str, a)], check=True, capture_output=True, text=True).stdout.split()]


def test_marches_whose_tiles_stay_empty_are_not_taken(rule):
    """Grids on which the march was measured slower than the two passes by 5 % or more do not take
    it, those on which it was faster by 10 % or more do (FP32; the single store's own rule by its size too)."""
    for shape, single, free in (((8, 8, 10000), False, False), ((33, 9, 2200), False, False), ((33, 33, 600), False, False),
                                ((16, 16, 4000), False, False), ((72, 72, 72), False, True), ((65, 65, 65), False, False),
                                ((40, 40, 40), False, False), ((96, 96, 96), True, True), ((80, 80, 80), True, True),
                                ((128, 128, 128), True, True), ((64, 64, 96), True, True), ((48, 48, 48), False, True)):
        assert rule(3, *shape, 16)[1:3] == [single, free], shape
    for nx, f32, f16 in ((16, False, False), (48, True, False), (96, True, True), (130, True, True), (260, True, True)):
        assert rule(2, nx, 4000, 1, 16)[2:] == [f32, f16], nx


def test_marches_fit_their_launch(rule):
    assert rule(3, 1, 524280, 1, 1)[0] and not rule(3, 1, 524281, 1, 1)[0]
    assert rule(3, 1, 1, 65535, 1)[0] and not rule(3, 1, 1, 65536, 1)[0] and rule(3, 1, 1, 65536, 2)[0]
    assert rule(2, 1, 65535, 1, 1)[0] and not rule(2, 1, 65536, 1, 1)[0]


def test_tiles_are_kept_for_fixed_faces(rule):
    """16-bit and FP32 grids with fixed-state faces ran on tiles up to some 724^2 nodes, which is where
    the march (with its tests of the faces) begins to win; without such faces it does from four tiles an SM on."""
    march, tile = 0, 1
    for shape, fixed, free in (((300, 500), tile, march), ((512, 512), tile, march), ((724, 724), tile, march),
                               ((1024, 1024), march, march), ((500, 300), tile, tile)):
        assert rule(-1, *shape, 1, 0, 1) == [fixed] and rule(-1, *shape, 1, 0, 0) == [free], shape


def test_small_launches_spread_over_the_sms_of_the_device(rule):
    """As many CTAs to an SM as all SMs need, whatever the device's number of them."""
    for sms in (76, 132, 148, 152, 160):
        for ctas in (1, sms, sms + 1, 2 * sms, 5 * sms - 1, 8 * sms, 8 * sms + 1):
            for stat in (0, 10240):
                k = -(-ctas // sms)
                assert rule(-9, ctas, sms, stat, 0) == [k if k <= 8 else 0], (sms, ctas, stat)
