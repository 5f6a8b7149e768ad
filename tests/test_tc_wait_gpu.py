"""A bounded wait that runs out in the radix-16 tensor-core kernel (every segment
length but 4096, which test_faults_gpu covers: another kernel).  As there:
OLS_TC_WAIT_NEVER=1 points the in-loop waits at an mbarrier nothing arrives on
and OLS_TC_WAIT_LIMIT=4 keeps them short; the kernel records the failure, drains
what it issued, releases its tensor memory and returns, and the next plan's
results are right."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1910_01972_gb300 import Plan, _native
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu
BOUND = {_native.OLS_FLAG_TC_FP16SPLIT: 2e-6, _native.OLS_FLAG_TC_BF16SPLIT: 3e-5}


# blocks of 128 threads (several segments, one segment) and of 512
@pytest.mark.parametrize("N,M", [(256, 33), (2048, 200), (8192, 700)])
@pytest.mark.parametrize("flag", list(BOUND))
def test_wait_runs_out(N, M, flag, monkeypatch):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    g = np.random.Generator(np.random.PCG64(N + flag))
    s, h = synth.signal(g, 60_000), synth.filters(g, 5, M)
    sd, hd = torch.from_numpy(s).cuda(), torch.from_numpy(h).cuda()
    monkeypatch.setenv("OLS_TC_WAIT_LIMIT", "4")
    monkeypatch.setenv("OLS_TC_WAIT_NEVER", "1")
    plan = Plan(M, 5, N, flags=flag)
    monkeypatch.delenv("OLS_TC_WAIT_LIMIT")
    monkeypatch.delenv("OLS_TC_WAIT_NEVER")
    plan.set_filters(hd)
    plan.convolve(sd)
    torch.cuda.synchronize()
    assert plan.status() != 0
    assert plan.status() == 0            # read and reset
    plan.close()
    plan = Plan(M, 5, N, flags=flag)
    plan.set_filters(hd)
    y = plan.convolve(sd).cpu().numpy()
    assert plan.status() == 0
    assert oracle.max_stream_rel_l2(y, oracle.conv(s, h)) <= BOUND[flag]
    plan.close()
