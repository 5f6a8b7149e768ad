"""FP32 results against 64 bits, as accurate as the plain form of the transforms
(a 16-point DFT per pass, one table-rounded twiddle per point, differences of the
output taken in the time domain) that the library's first kernels had.

Relative error over 8 filters of 400,000 samples (uniform signal, Gaussian taps,
complex FP32; real rows for the real form; derivative relative to itself): the
first column is that form's, measured on the same kind of inputs; the error of
so many outputs varies by less than 0.5% from seed to seed, and the bound leaves
1.5%.  Butterflies that take a - W b as 2 a - (a + W b) exceed it by 1 to 5%."""
import pytest
import torch

from paper_1910_01972_gb300 import Plan, _native
from paper_1910_01972_gb300 import build as _build

pytestmark = pytest.mark.gpu

#         N     M     plain  real   derivative   (1e-7)
FIGURES = [(256, 33, 1.45, 1.43, 1.485), (512, 65, 1.60, 1.59, 1.627), (1024, 129, 1.656, 1.637, 1.684),
           (2048, 257, 1.743, 1.722, 1.756), (4096, 513, 1.865, 1.848, 1.888), (8192, 1025, 1.99, 1.972, 2.01)]


def conv64(s, h):
    n, m = s.shape[0], h.shape[1]
    p = 1 << (n - 1).bit_length()
    S = torch.fft.fft(s.to(torch.complex128), p)
    return torch.stack([torch.fft.ifft(S * torch.fft.fft(r.to(torch.complex128), p))[m - 1:n] for r in h])


def rel(a, b):
    return float((a.to(b.dtype) - b).norm() / b.norm())


@pytest.mark.parametrize("N,M,plain,real,deriv", FIGURES)
def test_error_against_64_bits(N, M, plain, real, deriv):
    _build.build()
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    g = torch.Generator(device="cuda")
    g.manual_seed(N + 1)
    Ns, F = 400_000, 8
    s = torch.view_as_complex(torch.rand((Ns, 2), generator=g, device="cuda") * 2 - 1)
    h = torch.view_as_complex(torch.randn((F, M, 2), generator=g, device="cuda", dtype=torch.float64))
    hr = (h.real / torch.linalg.vector_norm(h.real, dim=1, keepdim=True)).to(torch.float32).contiguous()
    h = (h / torch.linalg.vector_norm(h, dim=1, keepdim=True)).to(torch.complex64)
    sr = s.real.contiguous()
    p, q = Plan(M, F, N), Plan(M, F, N, _native.OLS_FLAG_R2R)
    p.set_filters(h)
    q.set_filters_real(hr)
    y = conv64(s, h)
    d = torch.cat([y[:, 1:2] - y[:, :1], (y[:, 2:] - y[:, :-2]) / 2, y[:, -1:] - y[:, -2:-1]], dim=1)
    errors = rel(p.convolve(s), y), rel(q.convolve_real(sr), conv64(sr, hr).real), rel(p.convolve_derivative(s), d)
    for e, figure in zip(errors, (plain, real, deriv)):
        assert e <= 1.015e-7 * figure, (errors, (plain, real, deriv))
    p.close()
    q.close()
