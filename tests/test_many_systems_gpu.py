"""Edges of the batched solve: the near-diagonal band at the smallest sizes, and batches of so many systems that the
refinement takes its smaller CTAs, with problems that share their synthesis tables and nodes."""
import numpy as np
import pytest

import fh_inputs as fi
import oracle as O
from paper_1807_02718_gb300 import fh as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [F.FH_FP64, F.FH_MIXED_TF32])
@pytest.mark.parametrize("N", [8, 10, 32, 34, 66])
def test_small_matrices_match_the_oracle(precision, N):
    """Entries within 2e-13 of the largest (the double-float entries' stated error)."""
    cur = fi.small_kite(J=4, W=3.0).curve
    om = np.array([0.0, 0.5, 1.0, 1.5])
    pr = F.Problem(0, precision)
    pr.discretize(cur, om, np.full(4, N, dtype=np.int32), 1.0, (1.0, 0.0))
    for j in (1, 3):
        A, _ = F.fh_assemble_matrix(pr.ctx, j, om[j], N)
        ref = O.cfie_matrix(cur, N // 2, om[j])
        assert np.max(np.abs(A - ref)) <= 2e-13 * np.max(np.abs(ref))
    pr.close()


@pytest.mark.parametrize("precision", [F.FH_MIXED_TF32, F.FH_MIXED_BF16])
def test_many_systems_equal_each_problem_alone(precision):
    """14 stars, 686 systems of 1 to 3 blocks of 32 rows and ragged last blocks: bit for bit the problem alone."""
    rng = np.random.default_rng(4)
    probs = []
    for q in range(14):
        cur, J = fi.random_star(rng), 50 - q % 2       # two table sets
        om = fi.frequency_mesh(J, 6.0 + 0.5 * q)
        N = np.sort(2 * rng.integers(16, 49, J)).astype(np.int32)
        N[J // 2:J // 2 + 19] = N[J // 2]              # runs of equal sizes longer than one set of copies
        probs.append((cur, om, np.sort(N), (np.cos(q), np.sin(q))))
    ctx = F.fh_create(0, precision)
    F.fh_discretize_batch(ctx, [p[0] for p in probs], [p[1] for p in probs], [p[2] for p in probs], ps=[p[3] for p in probs])
    assert F.fh_solve_frequencies(ctx).n_solves > 4 * 152
    a = fi.sample_signal(fi.pulse_train(5, n=2, span=10.0, fmin=1.0, fmax=4.0), -10.0, 0.02, 1500)
    x, T = fi.targets_on_circle(5, 2.5), np.linspace(0.0, 40.0, 9)
    for q in (0, 1, 12, 13):
        cur, om, N, pdir = probs[q]
        F.fh_window_spectra_p(ctx, q, a, -10.0, 0.02)
        alone = F.Problem(0, precision)
        alone.discretize(cur, om, N, 1.0, pdir)
        alone.solve()
        alone.window_spectra(a, -10.0, 0.02)
        for j in range(1, len(om)):
            assert np.array_equal(F.fh_get_density_p(ctx, q, j, int(N[j])), F.fh_get_density(alone.ctx, j, int(N[j])))
        assert np.array_equal(F.fh_sample_p(ctx, q, x, T), alone.sample(x, T))
        alone.close()
    F.fh_destroy(ctx)


@pytest.mark.parametrize("omega", [0.9, 7.0, 61.0])
def test_fp64_fields_over_the_argument_range(omega):
    """FP64 target fields of a random density with kappa r from below 8 to past 1e4, the first and last intervals of
    the Hankel polynomials among them, against the oracle: 1e-13 of the largest covers 64 sums and phases of 1e4
    (2^-53 1e4 = 1e-12 at the far targets, whose fields are the smallest)."""
    N = 64
    wl = fi.circle_gauss(J=2, W=omega, N=N, n_x=3, n_T=4)
    rng = np.random.default_rng(3)
    psi = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    d = np.concatenate([np.geomspace(7.9, 2e4, 200) / omega, 8.0 / np.sqrt(np.arange(1, 33) / 32.0) / omega])
    d = 1.5 + d[d > 0.2]
    x = np.stack([d * np.cos(0.3), d * np.sin(0.3)], axis=1)
    pr = F.Problem(0, F.FH_FP64)
    pr.discretize(wl.curve, wl.omega, np.full(2, N, dtype=np.int32), 1.0, wl.p)
    F.fh_set_densities(pr.ctx, psi)
    pr.window_spectra(wl.a, wl.t0, wl.dt, wl.H)
    pr.sample(x, np.array([1.0]))
    V = F.fh_get_target_field(pr.ctx, len(x), 2)[:, 1]
    ref = O.target_field(wl.curve, N // 2, omega, psi, x, 1.0)
    near = omega * d < 100.0
    if near.any():
        assert np.max(np.abs(V - ref)[near]) <= 1e-13 * np.max(np.abs(ref))
    assert np.max(np.abs(V - ref)) <= 1e-12 * np.max(np.abs(ref))
    pr.close()
