"""Ids that warps claim ahead (GPU): CTAs whose warps meet for their last trajectories give back what
their reservoirs hold.  Stop-rule requests of trajectories of a few to a hundred blocks, alone and of two
kinds at once: warps claim ahead, the hand-out limit is passed and raised again and again, and CTAs are
always thin.  (A million trajectories of a few blocks with a 0.3 % rule: 3 to 9 warps per run hold ids
when their CTA meets.)  Every request completes, its prefix holds exactly the escape steps of the plain
kernel, and the bounds-checked build finds no reservoir after the meeting, nor a warp that waits for a
meeting nobody called when CTAs start a launch with nothing left to claim."""
import os
import subprocess
import sys

import pytest

import workloads

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = 1_000_003
OVER = workloads.scaled(workloads.overdamped_sweep(n_traj=1)[11], max_steps=10**6, stop_block=64, stop_rse=0.003)
BLOCKS = workloads.scaled(OVER, D=5.0, dt=0.05)
LONGER = workloads.scaled(OVER, dt=0.0125)
UNDER = workloads.scaled(workloads.plain_constant_tilt(), D=1.0, dt=0.05, precision="fp32", max_steps=3000,
                         stop_block=100, stop_rse=0.003)


def run_requests(problems, chunk, seeds):
    import paper_1802_05065_gb300 as m
    from paper_1802_05065_gb300 import api
    for seed in seeds:
        with m.Engine(0, chunk_steps=chunk) as eng:
            ids = [eng.submit(m.params_from(d, keep_per_traj=1), N, seed) for d in problems]
            for rid, d in zip(ids, problems):
                used = eng.wait(rid, 60.0).n_used
                k = eng.per_traj_steps(rid, used)
                assert used < N and (k == api.run_plain(d, used, seed).cpu().numpy()).all(), (chunk, seed)
            assert eng.counters()["check_flags"] == 0


@pytest.mark.parametrize("chunk", [1024, 4096, 16384])
@pytest.mark.parametrize("problems", [[BLOCKS], [UNDER], [BLOCKS, UNDER], [BLOCKS, LONGER]],
                         ids=["blocks", "underdamped", "two kinds", "two lengths"])
def test_every_id_of_the_prefix(problems, chunk):
    run_requests(problems, chunk, range(6))


@pytest.mark.parametrize("problem,chunks", [("BLOCKS", (1024, 4096, 16384)), ("LONGER", (64, 256, 1024))])
def test_checked_build(problem, chunks):
    from paper_1802_05065_gb300 import build as b
    b.build()
    code = f"""from tests.test_gpu_handout import *
for chunk in {chunks}: run_requests([{problem}], chunk, (1, 2, 3))"""
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=ROOT, timeout=900,
                       env=dict(os.environ, FPT_LIBRARY=b.LIB_CHECK))
    assert p.returncode == 0, p.stderr[-3000:]
