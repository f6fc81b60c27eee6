"""The FP64 kernel at the edges of its rounds and groups (GPU): trajectory counts around one lane
group, one group per SM and the lanes in flight, step budgets around a round of 64 steps, both
models and integrators, ramped bias, other sin amplitudes and thresholds of either sign."""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

OVER = workloads.scaled(workloads.overdamped_sweep(n_traj=1)[11], dt=0.05, precision="fp64",
                        max_steps=150)
UNDER = workloads.scaled(workloads.plain_constant_tilt(), D=0.5, dt=0.05, max_steps=150)


def _agree(d, n, seed, traj0=0):
    """Share of ids whose escape step is the oracle's.  A run is a few hundred steps, so a last-bit
    difference of a library function (1e-16, grown by at most e^10 over the run) moves a crossing
    with a probability of about 1e-10 per trajectory."""
    from paper_1802_05065_gb300 import api
    g = api.run_plain(d, n, seed, traj0=traj0).cpu().numpy()
    assert g.shape == (n,)
    ids = np.arange(n) if n <= 3000 else np.unique(np.concatenate(
        [np.arange(700), np.random.default_rng(n).integers(0, n, 1500), np.arange(n - 700, n)]))
    r = oracle.run_ids(oracle.params_from(d), seed, ids + traj0)
    return np.mean(g[ids] == np.asarray(r)), (g >= 0).mean()


@pytest.mark.parametrize("n", [1, 31, 33, 152 * 32 - 1, 152 * 32 + 1, 152 * 64 + 3, 152 * 128, 152 * 128 + 1, 50001])
def test_counts(n):
    same, esc = _agree(OVER, n, 11 + n)
    assert same >= 0.999 and (n < 1000 or 0.02 < esc < 0.9)


@pytest.mark.parametrize("cap", [1, 3, 4, 63, 64, 65, 128, 257])
def test_step_budgets(cap):
    same, _ = _agree(workloads.scaled(UNDER, max_steps=cap), 500, 5)
    assert same == 1.0


@pytest.mark.parametrize("over", [
    dict(integrator="heun"), dict(nu=0.05), dict(nu=0.05, integrator="heun"), dict(sin_amp=0.7),
    dict(sin_amp=0.0, nu=-0.01), dict(sin_amp=0.7, integrator="heun"),
    dict(threshold=0.0, threshold_mode="absolute", phi0=-1.0),
    dict(threshold=-0.5, threshold_mode="absolute", phi0=-2.0)])
@pytest.mark.parametrize("base", [OVER, UNDER], ids=["overdamped", "underdamped"])
def test_options(base, over):
    same, esc = _agree(workloads.scaled(base, **over), 2000, 77, traj0=2**32 - 100)
    assert same >= 0.999 and esc > 0.0


@pytest.mark.parametrize("over", [dict(), dict(integrator="heun"), dict(nu=0.05), dict(nu=0.05, integrator="heun"),
                                  dict(sin_amp=0.7), dict(max_steps=29)])
@pytest.mark.parametrize("n", [152 * 32 + 7, 152 * 64 - 1, 152 * 70])
def test_underdamped_pairs(over, n):
    """Two groups per CTA, each integrated by two warps, and three groups, by one each."""
    same, _ = _agree(workloads.scaled(UNDER, **over), n, 9)
    assert same >= 0.999
