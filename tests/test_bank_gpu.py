"""The bank kernel's work sharing and block sizes, and the derivative in the
frequency domain, against the FP64 oracle.

Shapes sit where the schedule can go wrong: fewer steps (blocks of segments x
filters) than resident CTAs, one filter, shares that begin and end inside a
segment's filters, idle slots in the last block, both block sizes.  Bounds are
those of the parity tests: 2e-6 relative L2 (FP32 path), the derivative's error
relative to the norm of y.
"""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1910_01972_gb300 import Plan, _native
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu
TOL = 2e-6


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")


def inputs(seed, Ns, F, M, real=False):
    g = np.random.Generator(np.random.PCG64(seed))
    if real:
        return synth.real_signal(g, Ns), synth.real_filters(g, F, M)
    return synth.signal(g, Ns), synth.filters(g, F, M)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# (N, M, F, Ns): one step in all; one filter over many blocks; steps just below,
# at and above the CTAs of a 148 .. 152-SM device; the 256- and 512-thread rule
SHAPES = [
    (256, 33, 1, 300), (256, 33, 3, 40_000), (256, 17, 61, 9_000),
    (512, 65, 1, 60_000), (512, 65, 7, 30_011), (512, 200, 40, 12_345),
    (1024, 129, 1, 9_000), (1024, 129, 19, 20_001), (2048, 257, 1, 40_000),
    (2048, 257, 61, 9_001), (2048, 257, 5, 61_000), (4096, 513, 1, 20_000),
    (4096, 513, 37, 15_000), (8192, 1025, 2, 40_000), (8192, 1025, 45, 9_000),
]


@pytest.mark.parametrize("N,M,F,Ns", SHAPES)
def test_schedule_against_oracle(N, M, F, Ns):
    s, h = inputs(N + M + F, Ns, F, M)
    plan = Plan(M, F, N)
    plan.set_filters(dev(h))
    y = plan.convolve(dev(s)).cpu().numpy()
    ref = oracle.conv(s, h)
    assert oracle.max_stream_rel_l2(y, ref, oracle.stream_scale(s, h, y.shape[1])) <= TOL
    plan.close()


@pytest.mark.parametrize("N,M,F", [(256, 33, 9), (512, 65, 9), (1024, 129, 9), (2048, 257, 9)])
def test_block_sizes_agree_bit_for_bit(N, M, F):
    """A segment's outputs do not depend on the block size or on where a CTA's
    share begins: a short signal (256-thread CTAs) equals the head of a long
    one (512-thread CTAs) in every segment they both hold whole."""
    L = N - M + 1
    s, h = inputs(N, 40 * L + M - 1, F, M)
    # the long signal: more than four steps of 512 threads per SM
    reps = 2 + (4 * 160 * (8192 // N) + F - 1) // F // 40
    long = np.concatenate([s] + [inputs(N + 1, 40 * L, F, M)[0]] * reps)
    plan = Plan(M, F, N)
    plan.set_filters(dev(h))
    a = plan.convolve(dev(s))
    b = plan.convolve(dev(long))
    assert torch.equal(a, b[:, :a.shape[1]])
    plan.close()


@pytest.mark.parametrize("N,M,F,Ns", [(256, 33, 5, 5_000), (512, 65, 33, 20_000), (2048, 257, 3, 30_000),
                                      (4096, 513, 7, 20_000)])
def test_real_schedule_against_oracle(N, M, F, Ns):
    s, h = inputs(N + F, Ns, F, M, real=True)
    plan = Plan(M, F, N, _native.OLS_FLAG_R2R)
    plan.set_filters_real(dev(h))
    y = plan.convolve_real(dev(s)).cpu().numpy()
    ref = oracle.conv_real(s, h)
    assert oracle.max_stream_rel_l2(y, ref, oracle.stream_scale(s, h, y.shape[1])) <= TOL
    plan.close()


@pytest.mark.parametrize("N,M", [(256, 33), (512, 65), (1024, 129), (2048, 257), (4096, 513), (8192, 1025)])
@pytest.mark.parametrize("extra", [2, 3, -1, 0, 1, 2 * 4096 + 5])
def test_derivative_ends(N, M, extra):
    """Two or three outputs in all, and a last segment of one output fewer
    than, exactly, and one more than a full one (the one-sided ends)."""
    step = N - M - 1
    nout = extra if extra in (2, 3) else 3 * step + extra
    s, h = inputs(N + extra + 7, nout + M - 1, 3, M)
    plan = Plan(M, 3, N)
    plan.set_filters(dev(h))
    d = plan.convolve_derivative(dev(s)).cpu().numpy()
    y = oracle.conv(s, h)
    ref = oracle.derivative(s, h)
    scale = oracle.stream_scale(s, h, nout)
    err = max(np.linalg.norm(d[f] - ref[f]) / max(np.linalg.norm(y[f]), scale[f]) for f in range(3))
    assert err <= TOL
    plan.close()


@pytest.mark.parametrize("N,M", [(256, 33), (512, 65), (1024, 129), (2048, 257)])
def test_smallest_blocks(N, M):
    """128-thread CTAs (at most one step each on 148 SMs or more) against the oracle, and bit for bit
    the head of a signal past that rule (256-thread CTAs), in each form."""
    F, L, per = 9, N - M + 1, 2048 // N                 # `per` segments to a 128-thread CTA
    s, h = inputs(N + 7, 60 * per * L + M - 1 - 5, F, M)          # 540 steps; the last segment ragged
    tail = inputs(N + 8, 20 * per * L, F, M)[0]                   # 720 in all
    plan = Plan(M, F, N)
    plan.set_filters(dev(h))
    a, b = plan.convolve(dev(s)), plan.convolve(dev(np.concatenate([s, tail])))
    whole = (60 * per - 1) * L
    assert torch.equal(a[:, :whole], b[:, :whole])
    y = a.cpu().numpy()
    assert oracle.max_stream_rel_l2(y, oracle.conv(s, h), oracle.stream_scale(s, h, y.shape[1])) <= TOL
    p, q = plan.convolve_power(dev(s)), plan.convolve_power(dev(np.concatenate([s, tail])))
    assert torch.equal(p[:, :whole], q[:, :whole])
    d, e = plan.convolve_derivative(dev(s)), plan.convolve_derivative(dev(np.concatenate([s, tail])))
    inner = (whole // (L - 2) - 1) * (L - 2)            # whole segments of the derivative in both signals
    assert torch.equal(d[:, :inner], e[:, :inner])
    plan.close()
