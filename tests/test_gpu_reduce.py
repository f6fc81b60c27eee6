"""The reduction of escape steps (GPU) against exact integer sums and the FP64 bins on the host: counts
around a load, a CTA's share and the grid, entries that start 8 but not 16 bytes aligned, bins in
shared and in global memory, no histogram, steps beyond 32 bits, and falling biases."""
import numpy as np
import pytest

import oracle
import workloads
from oracle import stats

pytestmark = pytest.mark.gpu

TIME = workloads.scaled(workloads.overdamped_sweep(n_traj=1)[11], hist_bins=100, hist_hi=60.0, max_steps=2**48)
BIAS = workloads.scaled(workloads.ramp_sweep(n_traj=1)[0], gamma0=0.1, hist_lo=0.15, hist_hi=0.9)


def _check(d, k, skip=0):
    import torch
    from paper_1802_05065_gb300 import api
    steps = torch.from_numpy(np.concatenate([np.full(skip, 7, np.int64), k])).cuda()[skip:]
    res, hist, s = api.reduce(d, steps)
    esc = [int(v) for v in k if v >= 0]
    assert (s.n_done, s.n_escaped) == (len(k), len(esc))
    assert s.s1_lo | s.s1_hi << 64 == sum(esc) and s.s2_lo | s.s2_hi << 64 == sum(v * v for v in esc)
    want = stats.summarize(oracle.params_from(d), k)
    assert (hist == want.hist).all() and (s.under, s.over) == (want.under, want.over)


def _steps(n, seed, mean=19000.0):
    rng = np.random.default_rng(seed)
    k = (rng.exponential(mean, n)).astype(np.int64) + 1
    k[rng.random(n) < 0.01] = -1
    return k


@pytest.mark.parametrize("skip", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 3, 1023, 4096, 4097, 152 * 4 * 4096 + 5])
def test_counts_and_alignment(n, skip):
    _check(TIME, _steps(n, n), skip)


@pytest.mark.parametrize("bins", [1, 1000, 8192, 8193, 1 << 20])
def test_bins(bins):
    _check(workloads.scaled(TIME, hist_bins=bins, hist_lo=0.5), _steps(100_001, bins))
    _check(workloads.scaled(BIAS, hist_bins=bins), _steps(50_001, bins, 5e6))


def test_long_steps_and_falling_bias():
    k = np.array([0, 1, 2**31, 2**32 - 1, 2**32, 2**32 + 1, 2**47, -1, 2**48], dtype=np.int64)
    _check(workloads.scaled(TIME, hist_hi=1e9), k)
    _check(workloads.scaled(BIAS, nu=-1e-6, hist_lo=-0.9, hist_hi=0.05), _steps(10_001, 3, 3e7))
    _check(workloads.scaled(BIAS, nu=0.0), _steps(1001, 4))
