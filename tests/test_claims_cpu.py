"""How many id blocks of a stop-rule request are handed out (CPU): always past the folded prefix, so
that a request whose rule is not met goes on to its last id; all of them when the expectation is not
a number or beyond 32 bits; and no fewer than expected.  Compiled with nvcc as host code."""
import subprocess

import numpy as np
import pytest

from tests.test_device_helpers_cpu import CSRC, _nvcc

PROGRAM = r"""
#include <cstdio>
#include "engine_dev.h"
int main() {
    double ids;
    unsigned block, prefix;
    unsigned long long n;
    while (std::scanf("%lf %u %u %llu", &ids, &block, &prefix, &n) == 4) {
        const unsigned b = fpt::claim_blocks_for(ids, block, prefix);
        std::printf("%u %llu\n", b, (unsigned long long)fpt::claim_end(n, block, b));
    }
    return 0;
}
"""


def test_claims(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not installed")
    src, exe = tmp_path / "c.cu", tmp_path / "c"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    rng = np.random.default_rng(1)
    cases = [(float("nan"), 4096, 7, 10**6), (float("inf"), 1, 0, 10), (0.0, 1, 0, 5), (0.0, 2**32 - 1, 0, 2**40),
             (1e4, 4096, 0, 2**18), (1e4, 4096, 3, 2**18), (1e30, 1, 2**32 - 1, 2**40)]
    for _ in range(3000):
        block = int(2 ** rng.uniform(0, 32))
        cases.append((float(10 ** rng.uniform(-2, 14)), min(block, 2**32 - 1),
                      int(rng.integers(0, 2**int(rng.integers(1, 33)))), int(2 ** rng.uniform(0, 40))))
    r = subprocess.run([str(exe)], input="\n".join("%r %d %d %d" % c for c in cases), capture_output=True, text=True)
    got = [tuple(map(int, l.split())) for l in r.stdout.splitlines()]
    assert len(got) == len(cases)
    for (ids, block, prefix, n), (b, end) in zip(cases, got):
        assert 0 < end <= n
        if b == 0:
            assert end == n
        else:
            assert prefix < b and b * block >= min(ids, 2.0**63) and end == min(n, b * block)
            assert b * block <= 1.25 * ids + 1.5 * prefix * block + prefix * block + 64 * 152 + 3 * block


SMS_PROGRAM = r"""
#include <cstdio>
#include "engine_dev.h"
int main() {
    for (int sms : {1, 76, 132, 148, 152, 160})
        for (unsigned prefix : {0u, 3u, 1000u})
            std::printf("%d %u %u\n", sms, prefix, fpt::claim_blocks_for(0.0, 64, prefix, sms));
    return 0;
}
"""


def test_look_ahead_follows_the_device(tmp_path):
    """Two warps per SM ahead of the folded prefix, whatever number of SMs the engine's device has."""
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not installed")
    src, exe = tmp_path / "s.cu", tmp_path / "s"
    src.write_text(SMS_PROGRAM)
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    lines = subprocess.run([str(exe)], capture_output=True, text=True).stdout.splitlines()
    assert len(lines) == 18
    for sms, prefix, blocks in (map(int, l.split()) for l in lines):
        assert max(64 * sms, 32 * prefix) <= 64 * (blocks - prefix) <= max(64 * sms, 32 * prefix) + 2 * 64
