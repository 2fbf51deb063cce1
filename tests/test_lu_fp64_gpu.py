"""FP64 batched LU over its sizes: systems of one panel, partial last panels, several strips, panels with more rows
than registers hold (N > 512), and couplings that force row exchanges, against numpy's solve of the assembled
matrices.

Tolerance: partial pivoting is backward stable, |dx|/|x| <~ cond N 2^-53 growth with cond < 1e3 here (second-kind
equation; at eta = 1000 omega the single layer dominates and cond stays below 1e4): 1e-11 covers N = 600."""
import numpy as np
import pytest

import fh_inputs as fi
from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("eta_scale", [1.0, 1000.0])
@pytest.mark.parametrize("sizes", [[8, 10, 16, 18, 30, 32, 34], [64, 62, 126, 130, 96], [510, 512, 514, 528, 600, 8],
                                   [258]])
def test_fp64_lu_sizes(sizes, eta_scale):
    cur = fi.kite()
    J = len(sizes) + 1
    omega = fi.frequency_mesh(J, 0.7 * len(sizes))
    N = np.array([64] + sizes, dtype=np.int32)
    eta = eta_scale * omega
    pr = F.Problem(0, F.FH_FP64)
    pr.discretize(cur, omega, N, 1.0, (0.6, 0.8))
    pr.solve(eta)
    for j in range(1, J):
        A, g = F.fh_assemble_matrix(pr.ctx, j, eta[j], int(N[j]))
        ref = np.linalg.solve(A, g)
        psi = F.fh_get_density(pr.ctx, j, int(N[j]))
        err = np.linalg.norm(psi - ref) / np.linalg.norm(ref)
        assert err < 1e-11, (int(N[j]), err)
    pr.close()
