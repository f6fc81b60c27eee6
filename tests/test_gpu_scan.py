"""The completion scan (GPU), 32 id blocks of a request at a time: sums, histogram and the stop rule's
prefix against exact arithmetic on the per-trajectory steps, for block counts around 32 and blocks of
one trajectory to more than the request has; and requests that reuse released buffers."""
import numpy as np
import pytest

import oracle
import workloads
from oracle import stats

pytestmark = pytest.mark.gpu

OVER = workloads.scaled(workloads.overdamped_sweep(n_traj=1)[11], dt=0.02, max_steps=2500, hist_bins=50,
                        hist_hi=60.0)


def _check(eng, m, d, n, seed):
    rid = eng.submit(m.params_from(d, keep_per_traj=1), n, seed)
    r = eng.wait(rid, 120.0)
    k = eng.per_traj_steps(rid, n)
    h, u, o = eng.histogram(rid, d["hist_bins"])
    s = eng.exact_sums(rid)
    eng.release(rid)
    p = oracle.params_from(d)
    used = n
    if d["stop_rse"] > 0:
        full = eng.submit(m.params_from(d, keep_per_traj=1, stop_rse=0.0), n, seed)
        eng.wait(full, 120.0)
        k = eng.per_traj_steps(full, n)
        eng.release(full)
        used = stats.stop_prefix(p, k, d["stop_rse"], d["stop_block"])
    assert r.n_used == used
    want = stats.summarize(p, k[:used])
    esc = [int(v) for v in k[:used] if v >= 0]
    assert (r.n_escaped, r.n_censored) == (len(esc), used - len(esc)) == (s.n_escaped, s.n_done - s.n_escaped)
    assert s.s1_lo | s.s1_hi << 64 == sum(esc) and s.s2_lo | s.s2_hi << 64 == sum(v * v for v in esc)
    assert list(h) == [int(c) for c in want.hist] and (u, o) == (want.under, want.over)
    return used


@pytest.mark.parametrize("block,n", [(1, 1), (1, 31), (1, 33), (7, 7 * 32), (7, 7 * 32 + 1), (64, 64 * 33 - 5),
                                     (100, 100_000), (4096, 5000), (1 << 20, 3000)])
def test_every_block(block, n):
    import paper_1802_05065_gb300 as m
    with m.Engine(0, chunk_steps=1024) as eng:
        assert _check(eng, m, workloads.scaled(OVER, stop_block=block), n, 10 + n) == n


@pytest.mark.parametrize("rse,block", [(0.3, 1), (0.1, 3), (0.05, 16), (0.03, 31), (0.02, 32), (0.01, 100), (1e-6, 512)])
def test_stop_rule(rse, block):
    import paper_1802_05065_gb300 as m
    with m.Engine(0, chunk_steps=1024) as eng:
        used = [_check(eng, m, workloads.scaled(OVER, stop_rse=rse, stop_block=block), 20_000, s) for s in (1, 2, 3)]
        assert all(u % block == 0 or u == 20_000 for u in used) and (rse < 1e-3) == (used[0] == 20_000)


def test_reused_buffers():
    """Sizes go up and down, so buffers of earlier requests with other layouts come back."""
    import paper_1802_05065_gb300 as m
    with m.Engine(0, chunk_steps=1024, max_requests=4) as eng:
        for i, (n, bins, block) in enumerate([(3000, 50, 64), (3000, 50, 64), (2500, 300, 100), (40_000, 20, 4096),
                                              (900, 1000, 7), (3001, 50, 64), (39_000, 1, 4096), (5, 2, 1)] * 3):
            _check(eng, m, workloads.scaled(OVER, hist_bins=bins, stop_block=block), n, i)


def test_stop_rule_hands_out_what_it_needs():
    """A request that stops early does not fill the lanes with ids past its result (the first hand-out
    is for 1.25 / rse^2 = 3125 or two warps per SM, 9728), and one whose rule is never met runs all."""
    import paper_1802_05065_gb300 as m
    for d, lo, hi in ((dict(stop_rse=0.02, stop_block=256), 1000, 25_000),
                      (dict(stop_rse=1e-5, stop_block=256), 200_000, 200_000)):
        with m.Engine(0, chunk_steps=1024) as eng:
            p = workloads.scaled(OVER, max_steps=10**6, **d)
            r = eng.wait(eng.submit(m.params_from(p), 200_000, 4), 120.0)
            c = eng.counters()
            assert lo <= r.n_used <= c["escapes"] + c["censored"] <= hi, (d, r.n_used, c)


def test_release_during_a_read():
    """One thread copies a finished request's steps while another releases it and runs the next, which
    would take its buffer: a copy that began gives the first request's steps."""
    import threading
    import time
    import paper_1802_05065_gb300 as m
    from paper_1802_05065_gb300 import api
    n, d = 500_001, workloads.scaled(OVER, max_steps=300)
    want = [api.run_plain(d, n, s).cpu().numpy() for s in range(2)]
    reads = 0
    with m.Engine(0, chunk_steps=4096) as eng:
        p = m.params_from(d, keep_per_traj=1)
        rid = eng.submit(p, n, 0)
        eng.wait(rid, 120.0)
        for i in range(40):
            got, begun = [], threading.Event()

            def read(rid=rid):
                begun.set()
                try:
                    got.append(eng.per_traj_steps(rid, n))
                except m.FptError as e:   # the release came first
                    got.append(e)
            t = threading.Thread(target=read)
            t.start()
            begun.wait()
            time.sleep(1e-4 * i)   # a copy takes ~1 ms: before, during and after it
            eng.release(rid)
            rid = eng.submit(p, n, (i + 1) % 2)
            eng.wait(rid, 120.0)
            t.join()
            if not isinstance(got[0], m.FptError):
                reads += 1
                assert (got[0] == want[i % 2]).all()
    assert reads > 0
