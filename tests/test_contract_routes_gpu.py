"""The contraction's routes (few outputs, FP64 tiles of 32 and 64, tensor cores) and the weights' column and group
edges against one another: a call with many times takes a large-size route, calls with few of the same targets and
times the others, and a time's weights do not depend on the other times of the call.

Tolerance: the same weights; sums of 2J products in FP64 (~2J 2^-53 of the sum of magnitudes) or, on the tensor
cores, ~2J 2^-49 of the largest row and column entries: 1e-12 relative to the row's norm covers 2J = 1026."""
import numpy as np
import pytest

import fh_inputs as fi
from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [F.FH_FP64, F.FH_MIXED_TF32])
@pytest.mark.parametrize("J,n_x", [(2, 70), (127, 333), (129, 130), (256, 65), (257, 64), (513, 33)])
def test_contraction_routes_agree(prec, J, n_x):
    wl = fi.circle_gauss(J=J, W=0.25 * (J - 1), N=64, n_x=n_x, n_T=8)
    rng = np.random.default_rng(J + n_x)
    V = rng.standard_normal((n_x, J)) + 1j * rng.standard_normal((n_x, J))
    n_T = (1 << 24) // (2 * J * n_x) + 37 if J > 2 else 300       # past the few-outputs route
    T = np.sort(rng.uniform(-5.0, 60.0, min(n_T, 2000)))
    pr = F.Problem(0, prec)
    pr.discretize(wl.curve, wl.omega, wl.N, wl.c, wl.p)
    pr.window_spectra(wl.a, wl.t0, wl.dt, wl.H)
    big = F.fh_synthesize(pr.ctx, V, T)
    assert np.all(np.isfinite(big))
    for sl in (slice(0, 1), slice(3, 8), slice(10, 27), slice(1, 66)):
        for nx in (1, 8, n_x):
            u = F.fh_synthesize(pr.ctx, V[:nx], T[sl])
            err = np.linalg.norm(u - big[:nx, sl]) / np.linalg.norm(big[:nx])
            assert err < 1e-12, (sl, nx, err)
    pr.close()
