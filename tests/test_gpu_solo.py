"""fpt_run_noalloc (GPU) at the edges of its CTAs' id ranges: escape steps, exact sums and histogram
equal those of the plain FP32 kernel and the host's statistics of its steps, for counts around a warp,
the packed groups, the lanes and beyond, every kind of step, one bin to the most it takes, ids above
2^32, accumulation into the outputs, and calls that overlap on two streams."""
import numpy as np
import pytest

import oracle
import workloads
from oracle import stats

pytestmark = pytest.mark.gpu

OVER = workloads.scaled(workloads.overdamped_sweep(n_traj=1)[11], dt=0.02, max_steps=3001, hist_hi=50.0)
UNDER = workloads.scaled(workloads.plain_constant_tilt(), D=0.08, dt=0.02, precision="fp32",
                         max_steps=20011, hist_hi=300.0)
RAMP = workloads.scaled(workloads.ramp_sweep(n_traj=1, rates=(2e-3,))[0])


class _Call:
    def __init__(self, d, n, seed):
        import torch
        self.d, self.n, self.seed = d, n, seed
        self.steps = torch.full((n,), -7, dtype=torch.int64, device="cuda")
        self.out = torch.zeros(8 + d["hist_bins"], dtype=torch.int64, device="cuda")

    def launch(self, stream=None):
        import paper_1802_05065_gb300 as m
        from paper_1802_05065_gb300 import api
        m.run_noalloc(m.params_from(self.d), self.n, self.seed, self.steps.data_ptr(), self.out.data_ptr(),
                      self.out.data_ptr() + 64, stream if stream is not None else api.current_stream())
        return self

    def check(self, times=1):
        from paper_1802_05065_gb300 import api
        want = api.run_plain(self.d, self.n, self.seed, traj0=self.d.get("traj_offset", 0)).cpu().numpy()
        assert (self.steps.cpu().numpy() == want).all()
        s = stats.summarize(oracle.params_from(self.d), want)
        got = [int(v) for v in self.out.cpu().numpy()]
        esc = [int(k) for k in want if k >= 0]
        s1, s2 = got[2] + (got[3] << 64), got[4] + (got[5] << 64)
        assert got[:2] == [times * self.n, times * len(esc)] and (s1, s2) == (times * sum(esc), times * sum(k * k for k in esc))
        assert got[6:8] == [times * s.under, times * s.over] and got[8:] == [times * int(c) for c in s.hist]


@pytest.mark.parametrize("n", [1, 31, 33, 152 * 32 + 1, 152 * 160, 152 * 160 + 1, 97280, 97281, 300007])
def test_counts(n):
    _Call(OVER, n, 3 + n).launch().check()


@pytest.mark.parametrize("d", [
    UNDER, RAMP, workloads.scaled(OVER, nu=1e-3), workloads.scaled(OVER, integrator="heun"),
    workloads.scaled(UNDER, integrator="heun", dt=0.05), workloads.scaled(RAMP, integrator="heun"),
    workloads.scaled(OVER, nu=1e-3, integrator="heun"), workloads.scaled(OVER, hist_bins=1),
    workloads.scaled(OVER, hist_bins=10240), workloads.scaled(OVER, traj_offset=2**33 - 7)])
def test_options(d):
    _Call(d, 30001, 5).launch().check()


def test_accumulates_and_overlaps():
    import torch
    a, b = _Call(OVER, 50001, 1), _Call(UNDER, 20001, 2)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        a.launch(s1.cuda_stream)
        b.launch(s2.cuda_stream)
    torch.cuda.synchronize()
    a.check(3)
    b.check(3)


CAPTURE = """
import torch
from tests.test_gpu_solo import *
from tests.test_gpu_solo import _Call
a = _Call(OVER, 50001, 4)
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):   # the process's first call of the library
    a.launch(torch.cuda.current_stream().cuda_stream)
for _ in range(3):
    g.replay()
torch.cuda.synchronize()
a.check(3)
"""


def test_first_call_inside_a_stream_capture():
    import os
    import subprocess
    import sys
    p = subprocess.run([sys.executable, "-c", CAPTURE], capture_output=True, text=True, timeout=600,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert p.returncode == 0, p.stderr[-3000:]
