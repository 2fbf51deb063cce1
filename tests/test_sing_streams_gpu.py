"""The split synthesis called on two streams at once: each call keeps its own graded mesh."""
import numpy as np
import pytest

from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


def cplx(rng, *sh):
    return rng.standard_normal(sh) + 1j * rng.standard_normal(sh)


def dev(z):
    import torch
    return torch.from_numpy(np.ascontiguousarray(z).view(np.float64).ravel()).cuda()


def test_two_streams_with_different_meshes():
    """A short call with another w_c runs while a long one is between its smooth and its singular weights.  Bit for
    bit the calls alone."""
    import torch
    rng = np.random.default_rng(2)
    J, W, K, n_x = 256, 40.0, 29, 3
    s, B, Bs, V, Vs = 15.0 * np.arange(K), cplx(rng, K, J), cplx(rng, K, 24), cplx(rng, J, n_x), cplx(rng, 24, n_x)
    d = [dev(v) for v in (s, B, Bs, V, Vs)]
    T = {5: dev(np.sort(rng.uniform(0.0, 400.0, 60000))), 7: dev(np.sort(rng.uniform(0.0, 400.0, 5)))}
    streams = {q: torch.cuda.Stream() for q in T}

    def call(j_c):
        u = torch.full((n_x * T[j_c].numel(),), float("nan"), device="cuda", dtype=torch.float64)
        streams[j_c].wait_stream(torch.cuda.current_stream())
        F.fh_synthesize_sing(J, W, j_c, *d, T[j_c], u, streams[j_c].cuda_stream)
        return u
    alone = {}
    for j_c in T:
        alone[j_c] = call(j_c)
        torch.cuda.synchronize()
    for rep in range(4):
        a = call(5)
        b = call(7)
        torch.cuda.synchronize()
        assert torch.equal(a, alone[5]), rep
        assert torch.equal(b, alone[7]), rep
