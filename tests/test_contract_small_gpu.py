"""The contraction of few outputs (up to 2^24 products, one launch) at the ends of its range: more times than a grid's
second dimension has tiles of 16, more targets than it has tiles of 8, and enough outputs for one frequency slice per
CTA, against calls of a few of the same targets and times.

Tolerance: the same weights; sums of 2J <= 128 products in FP64 in another order (2J 2^-53 of the sum of magnitudes,
1.4e-14), an order of magnitude of room for sums that cancel: 1e-12 of the row's norm."""
import numpy as np
import pytest

import fh_inputs as fi
from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [F.FH_FP64, F.FH_MIXED_TF32])
@pytest.mark.parametrize("J,n_x,n_T", [(2, 1, 65535 * 16 + 1), (2, 3, 65537 * 16 + 5), (2, 65536 * 8 + 3, 2), (64, 2500, 17)])
def test_many_times_or_targets(prec, J, n_x, n_T):
    assert 2 * J * n_x * n_T <= 1 << 24
    wl = fi.circle_gauss(J=J, W=0.25 * (J - 1), N=64, n_x=2, n_T=8)
    rng = np.random.default_rng(n_T)
    V = rng.standard_normal((n_x, J)) + 1j * rng.standard_normal((n_x, J))
    T = np.sort(rng.uniform(-5.0, 60.0, n_T))
    pr = F.Problem(0, prec)
    pr.discretize(wl.curve, wl.omega, wl.N, wl.c, wl.p)
    pr.window_spectra(wl.a, wl.t0, wl.dt, wl.H)
    u = F.fh_synthesize(pr.ctx, V, T)
    assert np.all(np.isfinite(u))
    for x in {0, n_x // 2, n_x - 1}:
        for t in {0, n_T // 2, n_T - 1}:
            xs, ts = slice(max(x - 9, 0), x + 1), slice(max(t - 20, 0), t + 1)
            few = F.fh_synthesize(pr.ctx, V[xs], T[ts])
            assert np.linalg.norm(few - u[xs, ts]) <= 1e-12 * np.linalg.norm(few)
    pr.close()
