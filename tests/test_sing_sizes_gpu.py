"""The split synthesis at many frequencies, on either side of what shared memory holds per time."""
import numpy as np
import pytest

from oracle import fh_sing as S
from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


def dev(z):
    import torch
    return torch.from_numpy(np.ascontiguousarray(z).view(np.float64).ravel()).cuda()


def reference(J, W, j_c, s, B, Bs, V, Vs, T):
    """synthesize_sing of the oracle with its coefficients by numpy's FFT (its DFT matrix has L^2 entries)."""
    om = np.linspace(0.0, W, J)
    wc, n = om[j_c], J - j_c
    A, delta, u = 0.5 * (W - wc), 0.5 * (W + wc), np.zeros((V.shape[0], T.size))
    for k in range(len(s)):
        for i in range(V.shape[0]):
            g = S.fc_extend(B[k, j_c:] * V[i, j_c:])
            L = g.size
            m = np.arange(-(L // 2), L // 2)
            P = L * (W - wc) / (n - 1)
            c = np.fft.fftshift(np.fft.fft(g)) / L * np.exp(1j * np.pi * (m * (n - 1) % (2 * L)) / L)
            tk = T - s[k]
            u[i] += (S.fourier_series_transform(c, A, P, delta, tk) + S.fcc_integral(Bs[k] * Vs[i], wc, tk)).real / np.pi
    return u


@pytest.mark.parametrize("n", [5105, 5107, 14001])
def test_many_frequencies(n):
    """Smooth spectra and fields (distances up to 3), times inside and far beyond the transform's period, more of them
    than one launch of the large sizes takes; 1e-9 of u: the operator's pairs carry 2^-48 and the continuation's
    entries reach 6e4."""
    import torch
    rng = np.random.default_rng(n)
    j_c, n_x, n_T = 4, 2, 650
    J, W = n + j_c, 0.02 * (n + j_c - 1)
    om = np.linspace(0.0, W, J)
    s = 15.0 * np.arange(2)
    spec = lambda w: np.stack([(1 + 0.5j * k) * np.exp(-0.5 * ((w - (0.3 + 0.1 * k) * W) / (0.2 * W)) ** 2) for k in range(2)])
    field = lambda w: np.stack([np.exp(1j * w * r) for r in (0.7, 2.9)])
    ws = F.fh_sing_frequencies(om[j_c])
    T = np.concatenate([rng.uniform(-5.0, 60.0, n_T - 50), rng.uniform(-2e3, 2e3, 50)])
    B, Bs, V, Vs = spec(om), spec(ws), field(om), field(ws)
    d_u = torch.full((n_x * n_T,), float("nan"), device="cuda", dtype=torch.float64)
    F.fh_synthesize_sing(J, W, j_c, dev(s), dev(B), dev(Bs), dev(V.T), dev(Vs.T), dev(T), d_u,
                         torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    u = d_u.cpu().numpy().reshape(n_x, n_T)
    pick = np.concatenate([np.arange(0, n_T, 37), np.arange(n_T - 60, n_T, 7)])
    ref = reference(J, W, j_c, s, B, Bs, V, Vs, T[pick])
    assert np.all(np.isfinite(u))
    err = np.linalg.norm(u[:, pick] - ref) / np.linalg.norm(ref)
    assert err < 1e-9, err
