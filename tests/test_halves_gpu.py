"""N = 8192 as two 4096-point halves where its index maps can go wrong: the
spectrum's storage order, the time-domain order of every form's output (ends,
both halves, one segment and several), peaks next to every edge of a warp and of
the halves, the batch beside plain calls; against the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1910_01972_gb300 import BatchPlan, Plan, _native, decode_candidates
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu
N, M, F = 8192, 700, 3


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_delta_filters_bit_exact():
    """Integer samples through delta filters come back exactly after rounding,
    at every position of a segment and of its ragged successor."""
    Ns = 2 * N + 1234
    n = np.arange(Ns)
    s = ((n % 509) + 1j * ((5 * n) % 509)).astype(np.complex64)
    h = np.zeros((3, 300), np.complex64)
    for f, d in enumerate((0, 123, 299)):
        h[f, d] = 1
    p = Plan(300, 3, N)
    p.set_filters(dev(h))
    y = p.convolve(dev(s)).cpu().numpy()
    for f, d in enumerate((0, 123, 299)):
        assert np.array_equal(np.round(y[f].real) + 1j * np.round(y[f].imag), s[299 - d:Ns - d])
    p.close()


@pytest.mark.parametrize("Ns", [M, 5000, N, N + 1, 30_000])
def test_forms_against_oracle(Ns):
    g = np.random.Generator(np.random.PCG64(Ns))
    s, h = synth.signal(g, Ns), synth.filters(g, F, M)
    p = Plan(M, F, N)
    p.set_filters(dev(h))
    y_ref = oracle.conv(s, h)
    scale = oracle.stream_scale(s, h, y_ref.shape[1])
    y = p.convolve(dev(s))
    assert oracle.max_stream_rel_l2(y.cpu().numpy(), y_ref, scale) <= 2e-6
    pw = p.convolve_power(dev(s)).cpu().numpy()
    assert np.max(np.linalg.norm(pw - oracle.power(s, h), axis=1)
                  / np.maximum(np.linalg.norm(oracle.power(s, h), axis=1), scale ** 2 / np.sqrt(pw.shape[1]))) <= 8e-6
    b = BatchPlan([Ns, Ns], [M, 33], [F, F], N=[N, 256])
    b.set_filters([dev(h), dev(synth.filters(g, F, 33))])
    assert torch.equal(b.convolve([dev(s), dev(s)])[0], y)
    sr, hr = synth.real_signal(g, Ns), synth.real_filters(g, F, M)
    r = Plan(M, F, N, _native.OLS_FLAG_R2R)
    r.set_filters_real(dev(hr))
    yr = oracle.conv_real(sr, hr)
    got = r.convolve_real(dev(sr)).cpu().numpy()
    assert oracle.max_stream_rel_l2(got, yr, oracle.stream_scale(sr, hr, yr.shape[1])) <= 2e-6
    for q in (p, b, r):
        q.close()


def test_peaks_at_every_position():
    """The peak rule applied to the kernel's own powers (as the power call gives
    them) marks the same set: neighbours across warps, registers and halves."""
    g = np.random.Generator(np.random.PCG64(5))
    s, h = synth.signal(g, 2 * N), synth.filters(g, F, M)
    p = Plan(M, F, N)
    p.set_filters(dev(h))
    pw = p.convolve_power(dev(s)).cpu().numpy()
    f, j, power = decode_candidates(*p.convolve_peaks(dev(s), 0.0, pw.size))
    got = np.zeros(pw.shape, bool)
    got[f, j] = True
    want = np.array([oracle.peak_mask(row[None], 0.0)[0] for row in pw])
    # segments of the two calls differ, and powers by rounding: a neighbour
    # within 1e-5 of the peak may decide differently
    pad = np.pad(pw, ((0, 0), (1, 1)), constant_values=-1)
    near = np.minimum(np.abs(pw - pad[:, :-2]), np.abs(pw - pad[:, 2:])) <= 1e-4 * np.maximum(pw, pw.mean())
    assert not np.any((got != want) & ~near)
    assert got.sum() > 1000
    p.close()
