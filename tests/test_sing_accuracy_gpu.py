"""The split synthesis on coarse meshes (the fields turn by one to two radians per frequency step), where the
continuation's entries of up to 6e4 do not cancel, against the same sums in extended precision.

Tolerance: the values that meet those entries are sums of 42 FP64 products, 2e-16 of a field's magnitude each; 31 of
them times 6e4 and the step over pi (0.2), three windows: 2e-11 of u, which the fields are of the size of, and half as
much again for the other roundings: 3e-11.  (In double-float pairs, 2^-48, they gave 4e-11 to 8e-11.)"""
import numpy as np
import pytest
from scipy.special import hankel1

import fh_inputs as fi
import oracle as O
from oracle import fh_sing as S
from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu

R, Z = np.longdouble, np.clongdouble
PI = R("3.14159265358979323846264338327950288")


def sinc(x):
    v = np.sin(PI * (x - 2 * np.rint(x / 2)))
    return np.where(x == 0, R(1), v / (PI * np.where(x == 0, R(1), x)))


def reference(J, W, j_c, s, B, Bs, V, Vs, T):
    At, Qt = (np.asarray(v, dtype=R) for v in S.fc_gram_table())
    n = J - j_c
    L, dw = n + 31, R(W) / (J - 1)
    wc = j_c * dw
    A, P, delta = (R(W) - wc) / 2, L * dw, (R(W) + wc) / 2
    m, l = np.arange(-(L // 2), L // 2), np.arange(L)
    D = np.exp(Z(-2j) * PI * (np.outer(m, l) % L).astype(R) / L) / L
    D = D * np.exp(Z(1j) * PI * ((m * (n - 1)) % (2 * L)).astype(R) / L)[:, None]
    u = np.zeros((V.shape[1], T.size), dtype=R)
    for k in range(len(s)):
        tk = T.astype(R) - R(s[k])
        row = 2 * A * sinc((2 * A / P) * (P / (2 * PI) * tk[:, None] - m[None, :].astype(R))) * np.exp(Z(-1j) * delta * tk)[:, None]
        for x in range(V.shape[1]):
            f = B[k, j_c:].astype(Z) * V[j_c:, x].astype(Z)
            g = np.concatenate([f, At @ (Qt.T @ f[-6:]) + (At @ (Qt.T @ f[:6][::-1]))[::-1]])
            u[x] += (row @ (D @ g)).real / PI + S.fcc_integral(Bs[k] * Vs[:, x], float(wc), T - s[k]).real / np.pi
    return u


@pytest.mark.parametrize("J,j_c,W", [(61, 4, 18.88), (35, 4, 27.14), (43, 4, 24.5), (27, 4, 25.88), (54, 5, 31.0)])
def test_coarse_meshes(J, j_c, W):
    import torch
    dev = lambda z: torch.from_numpy(np.ascontiguousarray(z).view(np.float64).ravel()).cuda()
    rng = np.random.default_rng(J)
    om = np.linspace(0.0, W, J)
    t0, dt = -10.0, 0.01
    sig = fi.pulse_train(J, n=12, span=60.0, fmin=W / 8, fmax=0.75 * W)
    a = fi.sample_signal(sig, t0, dt, int(np.ceil((sig.t_end - t0) / dt)) + 1)
    ws = F.fh_sing_frequencies(om[j_c])
    s, B = O.window_spectra(a, t0, dt, 10.0, om)
    _, Bs = O.window_spectra(a, t0, dt, 10.0, ws)
    x, src = 3.0 * np.exp(2j * np.pi * np.arange(3) / 3), rng.uniform(-0.5, 0.5, 3) + 1j * rng.uniform(-0.5, 0.5, 3)
    field = lambda w: sum(hankel1(0, np.outer(w, np.abs(x - z))) for z in src)
    V, Vs = np.concatenate([np.ones((1, 3)), field(om[1:])]), field(ws)
    T = np.sort(np.concatenate([rng.uniform(0.0, 90.0, 100), rng.uniform(0.0, 1000.0, 20)]))
    d_u = torch.full((3 * T.size,), float("nan"), device="cuda", dtype=torch.float64)
    F.fh_synthesize_sing(J, W, j_c, dev(s), dev(B), dev(Bs), dev(V), dev(Vs), dev(T), d_u,
                         torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    u = d_u.cpu().numpy().reshape(3, T.size)
    ref = reference(J, W, j_c, s, B, Bs, V, Vs, T)
    err = float(np.linalg.norm(u - ref.astype(np.float64)) / np.linalg.norm(ref.astype(np.float64)))
    assert err < 3e-11, err
