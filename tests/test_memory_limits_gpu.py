"""Calls that ask for more device memory than there is: refused with FH_ENOMEM, and nothing that they released is used
afterwards."""
import ctypes as C

import numpy as np
import pytest

import fh_inputs as fi
from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [F.FH_FP64, F.FH_MIXED_BF16])
def test_resident_fields_after_a_refused_sample(precision):
    """2e9 targets need 16 J 2e9 = 512 GB of fields: the resident ones went for them."""
    import torch
    wl = fi.circle_gauss(J=16, W=4.0, N=64, n_x=5, n_T=8)
    pr = F.Problem(0, precision)
    pr.discretize(wl.curve, wl.omega, wl.N, wl.c, wl.p)
    pr.solve()
    pr.window_spectra(wl.a, wl.t0, wl.dt, wl.H)
    T = np.linspace(0.0, 30.0, 7)
    u = pr.sample(wl.x, T)
    assert np.array_equal(F.fh_resample_p(pr.ctx, 0, T, wl.n_x), u)
    d = torch.zeros(16, device="cuda", dtype=torch.float64)   # never read: the call ends at the allocation
    ptr = C.c_void_p(d.data_ptr())
    st = F.load_library().fh_sample_p_dev(pr.ctx, 0, ptr, 2000000000, ptr, 1, ptr)
    assert st == F.FH_ENOMEM
    with pytest.raises(F.FHError) as e:
        F.fh_resample_p(pr.ctx, 0, T, wl.n_x)
    assert e.value.status == F.FH_ESTATE
    assert np.array_equal(pr.sample(wl.x, T), u)
    assert np.array_equal(F.fh_resample_p(pr.ctx, 0, T, wl.n_x), u)
    pr.close()
