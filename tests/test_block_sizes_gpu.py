"""The bank kernel's three block sizes give the same bits: one signal per size,
its length taken from the device's SM count and the rule of the dispatch
(128-thread CTAs while they leave each at most one step, four per SM; 256 under
four steps of 512 threads per SM; else 512), compared in every whole segment
that two of them share, and each with the oracle (2e-6 relative L2)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1910_01972_gb300 import Plan
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu


def block_of(nseg, F, N, sms):
    """The rule, restated: threads per CTA for nseg segments of F filters."""
    T = N // 16
    steps = {b: -(-nseg // (b // T)) * F for b in (128, 512)}
    return 128 if steps[128] <= 4 * sms else 256 if steps[512] < 4 * sms else 512


@pytest.mark.parametrize("N,M", [(256, 33), (512, 65), (1024, 129), (2048, 257)])
def test_three_block_sizes(N, M):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    F, L, T = 16, N - M + 1, N // 16
    per = {128: 128 // T, 512: 512 // T}                       # segments per CTA
    # the last length of the first rule, one between, the first of the third (each with a ragged last segment)
    nseg = [4 * sms // F * per[128], (4 * sms // F - 2) * per[512], -(-4 * sms // F) * per[512] + 3]
    assert [block_of(n, F, N, sms) for n in nseg] == [128, 256, 512]
    g = np.random.Generator(np.random.PCG64(N))
    s, h = synth.signal(g, nseg[2] * L + M - 1 - 5), synth.filters(g, F, M)
    plan = Plan(M, F, N)
    plan.set_filters(torch.from_numpy(h).cuda())
    sd = torch.from_numpy(s).cuda()
    ys = [plan.convolve(sd[:n * L + M - 1 - 5].contiguous()) for n in nseg]
    for n, y in zip(nseg[:2], ys):
        whole = (n - 1) * L
        assert torch.equal(y[:, :whole], ys[2][:, :whole])
    for y in ys:
        n = y.shape[1]
        for f in (0, F - 1):
            ref = oracle.conv(s[:n + M - 1], h[f:f + 1])
            assert oracle.max_stream_rel_l2(y[f:f + 1].cpu().numpy(), ref) <= 2e-6
    plan.close()


@pytest.mark.parametrize("M,F", [(513, 4), (513, 9), (4096, 4)])
def test_block_sizes_at_4096(M, F):
    """N = 4096: 512-thread CTAs from four steps per SM and four spectra on, else 256."""
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N, L = 4096, 4096 - M + 1
    short, long = 2 * ((4 * sms - 1) // F), 2 * -(-4 * sms // F) + 1        # segments; steps = ceil(n / 2) F
    assert -(-short // 2) * F < 4 * sms <= -(-long // 2) * F
    g = np.random.Generator(np.random.PCG64(M + F))
    s, h = synth.signal(g, long * L + M - 1), synth.filters(g, F, M)
    plan = Plan(M, F, N)
    plan.set_filters(torch.from_numpy(h).cuda())
    sd = torch.from_numpy(s).cuda()
    part = sd[:short * L + M - 1].contiguous()
    for call in (plan.convolve, plan.convolve_power):
        a, b = call(part), call(sd)
        assert torch.equal(a, b[:, :a.shape[1]])
    y = plan.convolve(sd)[F - 1:].cpu().numpy()
    assert oracle.max_stream_rel_l2(y, oracle.conv(s, h[F - 1:])) <= 2e-6
    plan.close()
