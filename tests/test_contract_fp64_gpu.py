"""FP64 sums on the tensor cores (fh_set_tuning contract_tc = 1, the default) against the plain FP64 kernel
(contract_tc = 0) and, for the split synthesis, against calls too small for the slices.

Tolerance: both sum 2J products; plain FP64 within 2J 2^-53 and the slices within 2J 2^-53 of the balanced row and
column maxima, which random fields exceed the result by sqrt(2J): 1e-12 of a row's norm covers 2J = 1026.  Products
past 2^25 take the slices."""
import numpy as np
import pytest

import fh_inputs as fi
from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


def both(J, V, T):
    wl = fi.circle_gauss(J=J, W=0.25 * (J - 1), N=64, n_x=V.shape[0], n_T=8)
    out = []
    for tc in (1, 0):
        pr = F.Problem(0, F.FH_FP64)
        F.fh_set_tuning(pr.ctx, contract_tc=tc)
        pr.discretize(wl.curve, wl.omega, wl.N, wl.c, wl.p)
        pr.window_spectra(wl.a, wl.t0, wl.dt, wl.H)
        out.append(F.fh_synthesize(pr.ctx, V, T))
        pr.close()
    return out


def fields(J, n_x, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((n_x, J)) + 1j * rng.standard_normal((n_x, J))


# tiles of 128 x 64, K segments of 512, K chunks of 16 padded to 64
@pytest.mark.parametrize("J,n_x,n_T", [(16, 1100, 1000), (129, 128, 1024), (256, 129, 513), (257, 257, 320), (513, 130, 300)])
@pytest.mark.parametrize("spread", [0, 12])
def test_slices_match_plain_fp64(J, n_x, n_T, spread):
    assert 2 * J * n_x * n_T > 1 << 25
    V = fields(J, n_x, J)
    V *= 10.0 ** (-spread * np.arange(J)[::-1] / J)     # the largest fields where the signal's spectrum has decayed
    u, u0 = both(J, V, np.linspace(0.0, 60.0, n_T))
    assert np.all(np.isfinite(u))
    assert np.all(np.linalg.norm(u - u0, axis=1) <= 1e-12 * np.linalg.norm(u0, axis=1))


def test_infinities_and_nan_stay_in_their_rows():
    V = fields(128, 300, 1)
    V[7, 3], V[131, 100], V[299, 127] = np.nan, np.inf, 1e308 + 1e308j
    V[12] = 0.0
    u, u0 = both(128, V, np.linspace(0.0, 60.0, 500))
    assert np.array_equal(np.isfinite(u), np.isfinite(u0))
    assert np.all(u[12] == 0.0) and not np.any(np.isfinite(u[7])) and not np.any(np.isfinite(u[131]))
    rows = np.setdiff1d(np.arange(300), [7, 131, 299])
    assert np.linalg.norm(u[rows] - u0[rows]) <= 1e-12 * np.linalg.norm(u0[rows])


def test_split_synthesis_with_slices():
    import torch
    J, j_c, W, n_x, n_T = 70, 5, 14.0, 400, 900
    rng = np.random.default_rng(5)
    dev = lambda z: torch.from_numpy(np.ascontiguousarray(z).view(np.float64).ravel()).cuda()
    cplx = lambda *sh: rng.standard_normal(sh) + 1j * rng.standard_normal(sh)
    s, B, Bs = 15.0 * np.arange(3), cplx(3, J), cplx(3, 24)
    w = np.linspace(0.0, W, J)[:, None]
    V = np.exp(1j * w * rng.uniform(0.5, 3.0, n_x))      # fields are smooth in the frequency
    Vs = cplx(24, n_x)
    T = np.sort(rng.uniform(-5.0, 80.0, n_T))

    def call(nx, T):
        d_u = torch.full((nx * T.size,), float("nan"), device="cuda", dtype=torch.float64)
        F.fh_synthesize_sing(J, W, j_c, dev(s), dev(B), dev(Bs), dev(V[:, :nx]), dev(Vs[:, :nx]), dev(T), d_u,
                             torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return d_u.cpu().numpy().reshape(nx, T.size)
    big = call(n_x, T)
    assert np.all(np.isfinite(big))
    for nx, sl in ((1, slice(0, 900)), (130, slice(60, 70)), (400, slice(897, 900))):
        u = call(nx, T[sl])
        # the continuation's weights reach 6e4, and both sums round at that magnitude: 2J 2^-53 6e4 / sqrt(2J)
        assert np.linalg.norm(u - big[:nx, sl]) <= 1e-10 * np.linalg.norm(u)
