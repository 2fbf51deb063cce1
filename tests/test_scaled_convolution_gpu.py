"""GPU parity of fh_scaled_convolution's FFTs over their sizes: one line, columns and lines of every split, the
plain transform of a power-of-two length and the chirp one, one and several lines per CTA, against the formula of
eq. approx_conv_sum evaluated with torch's FFTs (phases reduced in extended precision).

Tolerance: the values are sums of unit-size rotations of FFT outputs; an FFT of 2^25 points is accurate to
~25 * 2^-53 of the row's norm, four of them follow one another, and the phases are exact to ~2^-52 pi: 1e-13
relative L2 leaves a factor of five."""
import math

import numpy as np
import pytest

from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


def phase(num, L):
    """e^{i pi num / L} for an extended-precision num."""
    import torch
    r = torch.from_numpy(np.fmod(num / np.longdouble(L), np.longdouble(2)).astype(np.float64)).cuda() * math.pi
    return torch.polar(torch.ones_like(r), r)


def frft(x, alpha):
    import torch
    L = x.shape[-1]
    n = 1 << math.ceil(math.log2(2 * L))
    sq = lambda k: np.longdouble(alpha) * k.astype(np.longdouble) ** 2
    ch, kern = phase(-sq(np.arange(L) - L // 2), L), phase(sq(np.arange(L)), L)
    f = torch.zeros(n, dtype=torch.complex128, device="cuda")
    f[:L] = kern
    f[n - L + 1:] = kern[1:].flip(0)
    return torch.fft.ifft(torch.fft.fft(x * ch, n=n) * torch.fft.fft(f))[..., :L] * ch


def reference(c, beta, gamma, n0, L, A, P):
    import torch
    batch, M = c.shape
    x = torch.zeros(batch, L, dtype=torch.complex128, device="cuda")
    x[:, L // 2 - M // 2:L // 2 + M // 2] = c
    q = np.arange(L) - L // 2
    b = torch.from_numpy(2 * A * np.sinc(2 * A / P * q)).cuda().to(torch.complex128)
    y = frft(x, gamma) * frft(b, 1.0) * phase(2 * np.longdouble(beta) * n0 * q.astype(np.longdouble), L)
    return frft(y, -beta) / L


# (L, M, batch, gamma): Nf = 8 .. 2^21 with every column size of the split, odd remainders, many short rows
SIZES = [(2, 2, 3, 1.0), (4, 2, 1, 1.3), (6, 4, 5, 1.0), (8, 8, 2, 1.0), (30, 10, 37, 0.7), (128, 40, 3, 1.3),
         (500, 500, 2, 1.0), (1024, 100, 5, 1.0), (2048, 64, 1, 0.9), (2050, 64, 2, 1.0), (4096, 300, 3, 1.0),
         (8192, 10, 2, 1.0), (10000, 1000, 2, 1.0), (16384, 2, 1, 0.99), (65536, 1000, 2, 1.0), (70000, 5000, 1, 1.0),
         (131072, 4096, 1, 1.0), (262146, 100, 1, 1.01), (600000, 4000, 1, 1.0)]


@pytest.mark.parametrize("L,M,batch,gamma", SIZES + [(1 << 22, 1000, 1, 1.0), ((1 << 22) + 2, 1000, 1, 1.0),
                                                     ((1 << 23) + 2, 1000, 1, 1.0)])
def test_scaled_convolution_sizes(L, M, batch, gamma):
    import torch
    g = torch.Generator(device="cuda").manual_seed(L + M)
    c = torch.view_as_complex(torch.randn(batch, M, 2, dtype=torch.float64, device="cuda", generator=g))
    beta, n0, A, P = 0.37, 17 - L // 3, 2.0, 5.5
    d = torch.full((2 * batch * L,), float("nan"), device="cuda", dtype=torch.float64)
    F.fh_scaled_convolution(torch.view_as_real(c).reshape(-1), M, beta, gamma, n0, L, A, P, d,
                            torch.cuda.current_stream().cuda_stream)
    ref = reference(c, beta, gamma, n0, L, A, P)
    got = torch.view_as_complex(d.view(batch, L, 2))
    err = float(torch.linalg.norm(got - ref) / torch.linalg.norm(ref))
    assert err < 1e-13, err
