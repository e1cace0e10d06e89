"""CPU checks of the segment planner (choose_segment in csrc/elbm_internal.h), which the
allocation-free step runs on every call: the lengths against the rule evaluated for every number of
segments, and the time a call takes on long grids."""
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
