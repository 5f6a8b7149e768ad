"""The N = 4096 tensor-core form (two radix-64 stages) where its schedule and
layout can go wrong: one filter, an odd number of segments (an idle half tile),
shares that begin inside a segment pair's filters, the shortest signal, every
output position of one segment; against the FP64 oracle.  Bounds as in
test_tc_gpu: 2e-6 (FP16), 3e-5 (BF16)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1910_01972_gb300 import Plan, _native
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu
BOUND = {_native.OLS_FLAG_TC_FP16SPLIT: 2e-6, _native.OLS_FLAG_TC_BF16SPLIT: 3e-5}


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("flag", list(BOUND))
@pytest.mark.parametrize("M,F,Ns", [(512, 1, 512), (512, 1, 4096), (100, 2, 4097), (1, 3, 4096), (513, 1, 60_000),
                                    (513, 61, 11_000), (4096, 3, 4100), (257, 200, 8_000)])
def test_parity(flag, M, F, Ns):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    g = np.random.Generator(np.random.PCG64(M + F + flag))
    s, h = synth.signal(g, Ns), synth.filters(g, F, M)
    p = Plan(M, F, 4096, flags=flag)
    p.set_filters(dev(h))
    y = p.convolve(dev(s))
    assert p.status() == 0
    ref = oracle.conv(s, h)
    assert oracle.max_stream_rel_l2(y.cpu().numpy(), ref, oracle.stream_scale(s, h, ref.shape[1])) <= BOUND[flag]
    # the spectra read back in natural order, and the stored-split input bit for bit
    H = p.spectra().cpu().numpy()
    Href = np.fft.fft(h.astype(np.complex128), 4096, axis=1) / 4096
    assert np.max(np.abs(H - Href)) <= 6e-8 * np.max(np.abs(Href))
    hi, lo = p.split_signal(dev(s))
    assert torch.equal(p.convolve_split(hi, lo), y)
    p.close()


@pytest.mark.parametrize("M,amplitude", [(512, 64.0), (4000, 64.0), (512, 2.0 ** -6), (4000, 2.0 ** -6)])
def test_range_of_a_matched_tone(M, amplitude):
    # a tone in its matched filter gathers a segment's energy in one bin: the largest 16-bit operands
    # an amplitude can give.  The range is the radix-16 form's, FP16 split, bound as above.
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    Ns, w = 20_000, 2.0 * np.pi * 37 / 4096
    s = (amplitude * np.exp(1j * w * np.arange(Ns))).astype(np.complex64)
    h = (np.exp(1j * w * np.arange(M)) / np.sqrt(M)).astype(np.complex64)[None]
    p = Plan(M, 1, 4096, flags=_native.OLS_FLAG_TC_FP16SPLIT)
    p.set_filters(dev(h))
    y = p.convolve(dev(s)).cpu().numpy()
    assert p.status() == 0
    assert oracle.rel_l2(y, oracle.conv(s, h)) <= BOUND[_native.OLS_FLAG_TC_FP16SPLIT]
    p.close()


# relative error (1e-6) of the radix-16 form on the same tones
FAINT = [(2.0 ** -10, 16, 9.32), (2.0 ** -10, 64, 4.95), (2.0 ** -10, 512, 2.62), (2.0 ** -10, 4000, 0.84),
         (2.0 ** -8, 16, 2.31), (2.0 ** -8, 512, 0.90)]


@pytest.mark.parametrize("amplitude,M,figure", FAINT)
def test_faint_matched_tone(amplitude, M, figure):
    """FP16 parts below 2^-14 lose bits: the operands between the stages must not lose more of a faint
    signal than those of the radix-16 form did.  Against the samples as split, so that the rounding of
    the split itself, the same for both, neither adds nor cancels."""
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = 2.0 * np.pi * 37 / 4096
    s = (amplitude * np.exp(1j * w * np.arange(3 * 4096))).astype(np.complex64)
    x = s.view(np.float32)
    hi = x.astype(np.float16).astype(np.float32)
    split = (hi + (x - hi).astype(np.float16).astype(np.float32)).view(np.complex64)
    h = (np.exp(1j * w * np.arange(M)) / np.sqrt(M)).astype(np.complex64)[None]
    p = Plan(M, 1, 4096, flags=_native.OLS_FLAG_TC_FP16SPLIT)
    p.set_filters(dev(h))
    y = p.convolve(dev(s)).cpu().numpy()
    assert p.status() == 0
    assert oracle.rel_l2(y, oracle.conv(split, h)) <= 1e-6 * figure
    p.close()
