"""The adjoint's two block sizes: signals of a few windows (small blocks) and
just past the rule's limits (large ones), against the FP64 oracle and within
the built-in scratch.  Bounds of the adjoint's parity tests: ds 2e-6, dh 1e-5."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1910_01972_gb300 import Plan, _native
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,F,windows", [
    (256, 33, 3, 1), (256, 33, 3, 9), (256, 33, 2, 33), (512, 65, 5, 5), (512, 65, 8, 17), (1024, 129, 4, 3),
    (1024, 129, 16, 129), (2048, 257, 3, 2), (2048, 257, 8, 5), (4096, 513, 2, 3), (8192, 1025, 2, 2),
])
def test_few_windows_against_oracle(N, M, F, windows):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    nout = windows * (N - M + 1) - 3
    g = np.random.Generator(np.random.PCG64(N + F + windows))
    s, h = synth.signal(g, nout + M - 1), synth.filters(g, F, M)
    gy = (g.normal(size=(F, nout)) + 1j * g.normal(size=(F, nout))).astype(np.complex64)
    plan = Plan(M, F, N)
    plan.set_filters(torch.from_numpy(h).cuda())
    assert plan.backward_workspace(s.size) <= _native.OLS_NOALLOC_SCRATCH_BYTES
    ds, dh = plan.convolve_backward(torch.from_numpy(s).cuda(), torch.from_numpy(gy).cuda())
    ds_ref, dh_ref = oracle.adjoint(s, h, gy)
    assert oracle.rel_l2(ds.cpu().numpy(), ds_ref) <= 2e-6
    assert oracle.max_stream_rel_l2(dh.cpu().numpy(), dh_ref) <= 1e-5
    plan.close()


@pytest.mark.parametrize("N,M,F,windows", [(2048, 2048, 2, 512), (512, 511, 6, 2432), (256, 255, 13, 4864)])
def test_scratch_still_takes_long_filters(N, M, F, windows):
    # edges (16 windows (M - 1) bytes) beside the spectra of every small block would exceed the
    # scratch; those of the large blocks fit it
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    plan = Plan(M, F, N)
    assert plan.backward_workspace(windows * (N - M + 1) + M - 1) <= _native.OLS_NOALLOC_SCRATCH_BYTES
    plan.close()
