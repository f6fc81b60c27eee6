"""The engine's last trajectories of a CTA (GPU): groups of an integrating warp and noise warps must
give exactly the escape steps of the plain FP32 kernel, for counts around a group and around what
the groups take on, launch lengths around a round and a chunk of noise, CTA sizes with one to five
groups and none, every kind of step, and several kinds in one engine."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

OVER = workloads.scaled(workloads.overdamped_sweep(n_traj=1)[11], dt=0.01, max_steps=10**6)
UNDER = workloads.scaled(workloads.plain_constant_tilt(), D=0.08, dt=0.02, precision="fp32",
                         max_steps=20011)
RAMP = workloads.scaled(workloads.ramp_sweep(n_traj=1, rates=(2e-3,))[0])
KINDS = [OVER, UNDER, RAMP, workloads.scaled(OVER, nu=1e-3), workloads.scaled(OVER, integrator="heun"),
         workloads.scaled(UNDER, integrator="heun", dt=0.05), workloads.scaled(RAMP, integrator="heun"),
         workloads.scaled(OVER, nu=1e-3, integrator="heun")]


def _run(reqs, **kw):
    import paper_1802_05065_gb300 as m
    out = []
    with m.Engine(0, **kw) as eng:
        ids = [eng.submit(m.params_from(d, keep_per_traj=1), n, s) for d, n, s in reqs]
        for rid, (d, n, s) in zip(ids, reqs):
            r = eng.wait(rid, 300.0)
            k = eng.per_traj_steps(rid, n)
            h, u, o = eng.histogram(rid, d["hist_bins"])
            assert r.n_used == n and sum(h) + u + o == (k >= 0).sum() == r.n_escaped
            out.append(k)
        assert eng.counters()["useful_steps"] == sum(
            int(np.where(k >= 0, k, d["max_steps"]).sum()) for k, (d, _, _) in zip(out, reqs))
    return out


def _plain(d, n, s):   # one trajectory per thread, no shared machinery
    from paper_1802_05065_gb300 import api
    return api.run_plain(d, n, s).cpu().numpy()


@pytest.mark.parametrize("d", KINDS, ids=lambda d: f"{d['model']}-{d['integrator']}-{d['nu']:g}")
@pytest.mark.parametrize("n", [1, 33, 152 * 32 * 4 + 17])
def test_every_kind(d, n):
    [k] = _run([(d, n, 90 + n)], chunk_steps=16384)
    assert (k == _plain(d, n, 90 + n)).all()


@pytest.mark.parametrize("chunk", [16, 48, 64, 144, 4096, 4112, 65536])
def test_launch_lengths(chunk):
    n = 4099 if chunk < 1000 else 152 * 160
    d = workloads.scaled(OVER, max_steps=2000) if chunk < 1000 else OVER
    [k] = _run([(d, n, 7)], chunk_steps=chunk)
    assert (k == _plain(d, n, 7)).all()


@pytest.mark.parametrize("threads", [128, 256, 288, 320, 416, 512, 640])
def test_cta_sizes(threads):
    [k] = _run([(OVER, 30011, 8)], chunk_steps=8192, threads_per_block=threads)
    assert (k == _plain(OVER, 30011, 8)).all()


@pytest.mark.parametrize("threads,ctas", [(32, 16), (64, 10), (96, 6), (128, 5), (256, 2), (640, 1)])
def test_ctas_per_sm(threads, ctas):
    """What registers (20 warps of 96) and static shared memory allow: the groups cost no CTA."""
    from paper_1802_05065_gb300 import _lib
    assert _lib.engine_occupancy(1, threads) == ctas


def test_kinds_mixed():
    reqs = [(d, 700 + 301 * i, 50 + i) for i, d in enumerate(KINDS)]
    for k, (d, n, s) in zip(_run(reqs, chunk_steps=4096), reqs):
        assert (k == _plain(d, n, s)).all()


@pytest.mark.parametrize("threads", [256, 640])
def test_full_ctas_thin_out(threads):
    """More trajectories than lanes, of two kinds: warps meet several times and go on with fewer."""
    reqs = [(OVER, 97280 + 77, 60), (UNDER, 60001, 61)]
    for k, (d, n, s) in zip(_run(reqs, chunk_steps=4096, threads_per_block=threads), reqs):
        assert (k == _plain(d, n, s)).all()


@pytest.mark.parametrize("kw", [dict(chunk_steps=4096), dict(chunk_steps=80), dict(chunk_steps=4096, traj_per_thread=2)],
                         ids=["4096", "80", "two per thread"])
@pytest.mark.parametrize("d", [
    workloads.scaled(OVER, dt=0.05), workloads.scaled(OVER, dt=0.2, max_steps=150, integrator="heun"),
    workloads.scaled(UNDER, D=1.0, dt=0.05, max_steps=333), workloads.scaled(OVER, D=5.0, dt=0.05)],
    ids=["380 steps", "heun", "censored", "a few blocks"])
def test_short_trajectories_wait_for_each_other(d, kw):
    """Escapes of several blocks are published together; launches end while some wait."""
    n = 150_001 if kw["chunk_steps"] > 100 else 9_001
    [k] = _run([(d, n, 5)], **kw)
    assert (k == _plain(d, n, 5)).all()
