"""The reduction's integer bin map against the FP64 formula that defines the bins (CPU): whenever the
map names a bin (or under / over), the formula names the same one, for time and bias outputs, rising,
falling and constant observables, ranges that start below, at and above the first step, one bin to
2^20, and steps on both sides of every bin's edge; and it leaves few steps of a usual request open.

Compiled with nvcc as host code; skipped when nvcc is not installed."""
import os
import subprocess

import numpy as np
import pytest

from tests.test_device_helpers_cpu import CSRC, ROOT, _nvcc

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include "internal.h"
using namespace fpt;
static int formula(const Decoded &d, uint64_t k) {
    const double x = observable(d, k);
    if (x < d.hist_lo) return -1;
    if (x >= d.hist_hi) return d.hist_bins;
    volatile double y = x - d.hist_lo;
    y = y * d.hist_inv_w;
    const int b = static_cast<int>(std::floor(y));
    return b < d.hist_bins ? b : d.hist_bins - 1;
}
int main() {
    int output, bins;
    double dt, gamma0, nu, lo, hi;
    std::mt19937_64 rng(1);
    while (std::scanf("%d %d %lf %lf %lf %lf %lf", &output, &bins, &dt, &gamma0, &nu, &lo, &hi) == 7) {
        fpt_params p{};
        p.model = FPT_OVERDAMPED; p.output = output; p.hist_bins = bins; p.dt = dt; p.gamma0 = gamma0;
        p.nu = nu; p.hist_lo = lo; p.hist_hi = hi; p.D = 0.1; p.sin_amp = 1; p.phi0 = 0; p.threshold = 1;
        p.max_steps = 1;
        Decoded d;
        std::string err;
        if (!decode(&p, &d, &err)) { std::printf("bad %s\n", err.c_str()); continue; }
        const BinMap m = bin_map(d);
        std::vector<uint64_t> ks;
        for (uint64_t k = 0; k < 70; ++k) ks.push_back(k);
        for (int s = 6; s < 63; ++s)
            for (int o = -2; o <= 2; ++o) ks.push_back((1ull << s) + o);
        const size_t plain = ks.size();
        const double per = 1.0 / (d.out_b * d.hist_inv_w), k0 = (lo - d.out_a) / d.out_b;
        for (int i = 0; i <= 4000; ++i) {
            const double j = bins <= 4000 ? i % (bins + 1) : std::floor(bins * (i / 4000.0));
            const double c = k0 + j * per;
            if (!(std::fabs(c) < 4e18)) continue;
            for (int o = -3; o <= 3; ++o)
                if (c + o >= 0) ks.push_back(static_cast<uint64_t>(c + o));
        }
        const size_t edges = ks.size();
        const double a = std::fmax(0, std::fmin(k0, k0 + bins * per)), b = std::fmax(k0, k0 + bins * per);
        long open = 0, wrong = 0;
        for (int i = 0; i < 20000; ++i) {
            const double c = a + (b - a) * 1.1 * (rng() >> 11) * 0x1p-53;
            if (c >= 0 && c < 4e18) ks.push_back(static_cast<uint64_t>(c));
        }
        for (size_t i = 0; i < ks.size(); ++i) {
            const int g = ks[i] >= m.k_over ? bins : ks[i] < m.k_under ? -1
                          : ks[i] >> 32 ? -2 : mapped_bin(m, static_cast<uint32_t>(ks[i]));
            if (g == -2) { if (i >= edges && !(ks[i] >> 32)) ++open; continue; }
            if (g != formula(d, ks[i])) ++wrong;
        }
        (void)plain;
        std::printf("%ld %f %d\n", wrong, ks.size() > edges ? double(open) / (ks.size() - edges) : 0.0, m.span > 0);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def compare(tmp_path_factory):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not installed")
    d = tmp_path_factory.mktemp("bin_map")
    src, exe = d / "map.cpp", d / "map"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I", CSRC, "-I",
                        os.path.join(ROOT, "include"), "-o", str(exe), str(src),
                        os.path.join(CSRC, "common.cpp")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]

    def run(cases):
        text = "\n".join("%d %d %.17g %.17g %.17g %.17g %.17g" % c for c in cases)
        r = subprocess.run([str(exe)], input=text, capture_output=True, text=True, timeout=300)
        out = [l.split() for l in r.stdout.splitlines()]
        assert r.returncode == 0 and len(out) == len(cases) and all(len(l) == 3 for l in out), r.stdout[:500]
        return [(int(w), float(o), int(u)) for w, o, u in out]
    return run


def test_usual_requests(compare):
    cases = [(0, 100, 1e-3, 0.9, 0.0, 0.0, 1e4), (0, 100, 0.005, 0.8, 0.0, 0.0, 5000.0),
             (0, 64, 0.005, 0.8, 0.0, 0.0, 800.0), (0, 1000, 1e-3, 0.5, 0.0, 3.0, 200.0),
             (1, 1000, 0.01, 0.0, 1e-5, 0.5, 1.0), (1, 1000, 0.01, 0.0, 1e-8, 0.5, 1.0),
             (1, 300, 0.01, 0.7, 1e-6, 0.6, 0.9), (0, 1 << 20, 1e-3, 0.9, 0.0, 0.0, 1e7),
             (0, 1, 1e-3, 0.9, 0.0, 0.0, 100.0), (0, 7, 1e-3, 0.9, 0.0, -5.0, 100.0)]
    for c, (wrong, left, used) in zip(cases, compare(cases)):
        x0, dx = (0.0, c[2]) if c[0] == 0 else (c[3], c[4] * c[2])
        below = (c[5] - x0) / dx < 2**32       # the map is for steps below 2^32
        assert wrong == 0 and used == below and left < 0.01, (c, wrong, left, used)


def test_random_and_extreme_requests(compare):
    rng = np.random.default_rng(5)
    cases = []
    for _ in range(400):
        out = int(rng.integers(2))
        bins = int(10 ** rng.uniform(0, 6.02))
        dt = float(10 ** rng.uniform(-5, 0))
        g = float(rng.uniform(-1, 1))
        nu = float(rng.choice([-1, 0, 1]) * 10 ** rng.uniform(-12, 1))
        lo = float(rng.choice([0.0, g, rng.uniform(-2, 2), 10 ** rng.uniform(-3, 6)]))
        cases.append((out, bins, dt, g, nu, lo, lo + float(10 ** rng.uniform(-9, 9))))
    cases += [(1, 10, 0.1, 0.5, 0.0, 0.0, 1.0), (1, 10, 0.1, 0.5, -1e-3, 0.0, 1.0),
              (0, 5, 1.0, 0.0, 0.0, 0.0, 5.0), (0, 10, 1.0, 0.0, 0.0, 0.5, 3.0),
              (0, 3, 1e-300, 0.0, 0.0, 0.0, 1e-290), (0, 3, 1e300, 0.0, 0.0, 0.0, 1e305)]
    got = compare(cases)
    assert [c for c, (wrong, _, _) in zip(cases, got) if wrong] == []
    assert sum(u for _, _, u in got) > 100
