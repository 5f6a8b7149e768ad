"""Two 16-thread segments share a warp at N = 256.  Their per-segment code may
branch apart (a full segment beside a ragged or an idle one, an end segment of
the derivative beside an inner one), while the tensor-memory accesses around it
are warp-wide (`.sync.aligned`) and want the whole warp: the warp has to meet
again in between.

Whether it does is a property of the source (a compiled kernel may happen to
reconverge by itself), so it is read there; the results of the mixed warps are
compared with the oracle on the GPU, bound 2e-6 relative L2 as in the parity
tests (the derivative's relative to the norm of y)."""
import os
import re

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1910_01972_gb300 import BatchPlan, Plan
from paper_1910_01972_gb300 import build as _build

N, M, F = 256, 33, 3
L = N - M + 1


def statements_after(call):
    """The statement that follows each `epi.template <call><...>(...)` in the kernels' sources."""
    out = []
    for name in sorted(os.listdir(_build.CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(_build.CSRC, name)).read())
        for m in re.finditer(r"epi\.template %s<[^;]*;\s*([^;]*;?)" % call, text):
            out.append((name, " ".join(m.group(1).split())))
    return out


@pytest.mark.parametrize("call", ["store", "spectrum"])
def test_warp_meets_after_per_segment_code(call):
    found = statements_after(call)
    assert found
    for name, nxt in found:
        assert nxt == "if constexpr (G::T < 32) __syncwarp();", (name, nxt)


def test_warp_meets_after_candidate_records():
    """Only the lanes with a candidate write a record."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(_build.CSRC, "ols_post.cu")).read())
    record = re.search(r"cand\[i\] = c;([\s}]*)(\w+\(\);)?", text)
    assert record and record.group(2) == "__syncwarp();"


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


# a full segment beside a ragged one, beside an idle one, and a ragged one beside an idle one
@pytest.mark.gpu
@pytest.mark.parametrize("per_n", [False, True])
@pytest.mark.parametrize("nout", [5 * L + 100, 7 * L, 6 * L + 1, 50])
def test_batch_with_mixed_warps(per_n, nout):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    g = np.random.Generator(np.random.PCG64(nout))
    Ns = [nout + M - 1, 3 * L + M + 6]
    ss, hs = [synth.signal(g, n) for n in Ns], [synth.filters(g, F, M) for _ in Ns]
    b = BatchPlan(Ns, [M, M], [F, F], N=[N, N], per_n=per_n)
    b.set_filters([dev(h) for h in hs])
    for s, h, y in zip(ss, hs, b.convolve([dev(s) for s in ss])):
        assert oracle.max_stream_rel_l2(y.cpu().numpy(), oracle.conv(s, h), oracle.stream_scale(s, h, y.shape[1])) <= 2e-6
    b.close()


# inner segments beside the first, the last (full or ragged) and an idle one
@pytest.mark.gpu
@pytest.mark.parametrize("nout", [2, L, 2 * (L - 2), 5 * (L - 2), 6 * (L - 2) + 1, 7 * (L - 2) - 1])
def test_derivative_with_mixed_warps(nout):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    g = np.random.Generator(np.random.PCG64(nout))
    s, h = synth.signal(g, nout + M - 1), synth.filters(g, F, M)
    p = Plan(M, F, N)
    p.set_filters(dev(h))
    d = p.convolve_derivative(dev(s)).cpu().numpy()
    y, ref, scale = oracle.conv(s, h), oracle.derivative(s, h), oracle.stream_scale(s, h, nout)
    assert max(np.linalg.norm(d[f] - ref[f]) / max(np.linalg.norm(y[f]), scale[f]) for f in range(F)) <= 2e-6
    p.close()
