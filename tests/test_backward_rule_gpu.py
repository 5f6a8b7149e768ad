"""The adjoint's block-size rule at its limits: with dh the small blocks end where
their partial spectra cost more than they save (a call past the limit takes the
large blocks, seen in its workspace), without dh at four per SM; the gradients on
both sides of a limit against the FP64 oracle (bounds of the adjoint's parity
tests: ds 2e-6, dh 1e-5)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1910_01972_gb300 import Plan
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu

#        N    M   F  small blocks per SM with dh, in quarters
RULE = [(256, 33, 1, 4), (256, 33, 3, 4), (256, 33, 4, 8), (256, 17, 16, 12), (512, 65, 1, 4), (512, 65, 2, 6),
        (512, 65, 4, 8), (1024, 129, 1, 3), (1024, 129, 4, 4), (2048, 257, 2, 6), (4096, 513, 1, 4)]


def windows(N, blocks):
    return blocks * (max(N // 16, 128) // (N // 16))


@pytest.mark.parametrize("N,M,F,quarters", RULE)
def test_blocks_at_the_limit(N, M, F, quarters):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    plan, spec = Plan(M, F, N), 8 * F * N

    def partial_spectra(nwin):
        Ns = nwin * (N - M + 1) + M - 1
        return plan.backward_workspace(Ns, False, True) // spec - 1       # and their sum

    at = quarters * sms // 4
    large = (256 if N == 1024 else 512) // (N // 16)
    assert partial_spectra(windows(N, at)) == at
    past = windows(N, at) + 1
    assert partial_spectra(past) == min(-(-past // large), (512 // (large * (N // 16))) * sms)
    plan.close()


@pytest.mark.parametrize("N,M,F,quarters", [RULE[0], RULE[7]])
@pytest.mark.parametrize("more", [0, 1])
def test_gradients_at_the_limit(N, M, F, quarters, more):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nout = (windows(N, quarters * sms // 4) + more) * (N - M + 1) - 3
    g = np.random.Generator(np.random.PCG64(N + more))
    s, h = synth.signal(g, nout + M - 1), synth.filters(g, F, M)
    gy = (g.normal(size=(F, nout)) + 1j * g.normal(size=(F, nout))).astype(np.complex64)
    plan = Plan(M, F, N)
    plan.set_filters(torch.from_numpy(h).cuda())
    sd, gd = torch.from_numpy(s).cuda(), torch.from_numpy(gy).cuda()
    ds, dh = plan.convolve_backward(sd, gd)
    ds_ref, dh_ref = oracle.adjoint(s, h, gy)
    assert oracle.rel_l2(ds.cpu().numpy(), ds_ref) <= 2e-6
    assert oracle.max_stream_rel_l2(dh.cpu().numpy(), dh_ref) <= 1e-5
    # without dh the blocks may be others; a window's transforms are the same
    assert torch.equal(plan.convolve_backward(sd, gd, want_dh=False)[0], ds)
    plan.close()
