"""Rounds of a CTA's last trajectories (CPU), compiled with nvcc as host code: walked with no packing in
between past 2^33 blocks, far beyond what an int counts, every round is a positive number of blocks, they
double up to a cap, and a bounded launch runs exactly its blocks."""
import subprocess

import pytest

from tests.test_device_helpers_cpu import CSRC, _nvcc

PROGRAM = r"""
#include <cstdio>
#include "engine_dev.h"
int main() {
    unsigned long long blocks, stop;
    while (std::scanf("%llu %llu", &blocks, &stop) == 2) {   // a launch of `blocks`, looked at up to `stop` of them
        unsigned long long done = 0, rounds = 0;
        unsigned most = fpt::kRoundBlocks;
        int least = 0x7FFFFFFF, longest = 0;
        while (done < stop && done < blocks) {
            const int r = fpt::round_blocks(blocks - done, most);
            least = r < least ? r : least;
            longest = r > longest ? r : longest;
            if (r <= 0) break;
            done += r;
            ++rounds;
            most = fpt::longer_round(most);
        }
        std::printf("%llu %llu %d %d\n", done, rounds, least, longest);
    }
    return 0;
}
"""


def test_rounds(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not installed")
    src, exe = tmp_path / "r.cu", tmp_path / "r"
    src.write_text(PROGRAM)
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    cases = [(2**64 - 1, 2**33), (2**44, 2**33), (2**32 + 7, 2**33), (2**20, 2**33), (1, 9), (255, 9999), (257, 9999)]
    r = subprocess.run([str(exe)], input="\n".join("%d %d" % c for c in cases), capture_output=True, text=True, timeout=60)
    got = [tuple(map(int, l.split())) for l in r.stdout.splitlines()]
    assert len(got) == len(cases)
    for (blocks, stop), (done, rounds, least, longest) in zip(cases, got):
        assert least >= 1 and longest <= 2**20
        assert done == blocks if blocks < stop else done >= stop
        assert rounds <= 13 + done // 2**20   # doubling from 256, then 2^20 each
