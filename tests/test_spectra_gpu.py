"""Filter spectra (FP64 residue FFTs) against numpy's FP64 FFT of the padded
filters, at the edges of the residue decomposition: one tap, the residue length
N/16 and one more, a full segment.  One rounding to FP32: 6e-8 relative."""
import numpy as np
import pytest
import torch

import synth
from paper_1910_01972_gb300 import Plan
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [256, 512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("where", ["one", "below", "above", "full"])
def test_spectra_edges(N, where):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    M = {"one": 1, "below": N // 16, "above": N // 16 + 1, "full": N}[where]
    g = np.random.Generator(np.random.PCG64(N + M))
    h = synth.filters(g, 3, M)
    plan = Plan(M, 3, N)
    plan.set_filters(torch.from_numpy(h).cuda())
    H = plan.spectra().cpu().numpy()
    ref = np.fft.fft(h.astype(np.complex128), N, axis=1) / N
    assert np.max(np.abs(H - ref)) <= 6e-8 * np.max(np.abs(ref))
    plan.close()
