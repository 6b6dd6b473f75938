"""Which rows of a reduced-precision half sweep are drawn in float pairs, and how exact either form is.

X is pinned to odd integers (prior precision 1e60), so the FP32 Gram sums and right-hand sides of the
W rows are exact and what is left is the draw's own rounding.  A W row has n < K observations and the
prior I, so tau sum x x^T leaves K - n pivots that lose all but 1 / (tau g) of their diagonal.

Tolerances, relative to |x|, with the condition number kappa: pairs 4 K 2^-44 kappa; FP64 rounds at
2^-53, in this draw and in the reference, about sqrt(K) times an entry: 8 sqrt(K) 2^-52 kappa."""
import time

import numpy as np
import pytest

from paper_1703_00734_gb300 import synth

pytestmark = pytest.mark.gpu
D = 130             # two full conditional blocks of rows and two rows


def _draw(K, tau, n, prec="fp32", prior=None, seed=0):
    """W after one sweep, the same from FP64 arithmetic, and the condition numbers."""
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(100 * K + seed)
    N = 3 * K
    col = np.repeat(np.arange(D), n)
    row = np.concatenate([rng.choice(N, k, replace=False) for k in n])
    muX = rng.choice([-3.0, -1.0, 1.0, 3.0], (N, K))
    y = rng.integers(-8, 9, len(row)).astype(np.float64)
    mu, Lam = (np.zeros((D, K)), np.broadcast_to(np.eye(K), (D, K, K)).copy()) if prior is None else prior
    m = bmf.BMF(N, D, row, col, y, K, tau, prec, order="none", center=False, X0=muX, W0=np.zeros((D, K)))
    m.set_prior(0, bmf.FACTOR_X, muX, np.broadcast_to(1e60 * np.eye(K), (N, K, K)).copy())
    m.set_prior(0, bmf.FACTOR_W, mu, Lam)
    dr = synth.sweep_draws([(N, D)], K, float(K), synth.rng_for(seed, 1))
    m.sweep(0, 1, dr)
    _, W, _ = m.get_state(0)
    m.close()
    z = dr[-D * K:].reshape(D, K)
    want, kappa = np.empty((D, K)), np.empty(D)
    for j in range(D):
        x, v = muX[row[col == j]], y[col == j]
        P = Lam[j] + tau * x.T @ x
        L = np.linalg.cholesky(P)
        want[j] = np.linalg.solve(L.T, np.linalg.solve(L, Lam[j] @ mu[j] + tau * x.T @ v) + z[j])
        kappa[j] = np.linalg.cond(P)
    return np.linalg.norm(W - want, axis=1) / np.linalg.norm(want, axis=1), kappa


KS = [9, 10, 12, 13, 16, 17, 24, 25, 32, 33, 48]


@pytest.mark.parametrize("K", KS)
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_pivots_that_keep_28_bits_are_a_pairs(K, prec):
    n = np.random.default_rng(K).integers(1, K, D)
    err, kappa = _draw(K, 2.0 ** 10, n, prec)           # tau g < 2^10 9 48 < 2^19
    assert (err <= 4 * K * 2.0 ** -44 * kappa).all(), (err / kappa).max()


@pytest.mark.parametrize("K", KS)
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_pivots_that_lose_more_are_fp64s(K, prec):
    """tau g from 2^24 on, among rows that stay in pairs: those without enough to lose, whose n of 0."""
    n = np.random.default_rng(K).integers(1, K, D)
    n[::3] = 0
    err, kappa = _draw(K, 2.0 ** 24, n, prec)
    lossy = n > 0
    assert (err[lossy] <= 8 * np.sqrt(K) * 2.0 ** -52 * kappa[lossy]).all(), (err / kappa)[lossy].max() * 2.0 ** 52
    assert (err[~lossy] <= 4 * K * 2.0 ** -44).all()


@pytest.mark.parametrize("K", KS)
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_rows_whose_terms_are_fp64s(K, prec):
    """Rows without observations, and rows whose sums are below 2^-16 of their prior in every diagonal
    entry (2^-32 9 48 here): the prior and the draw are FP64's and so is x.  Diagonal priors: about
    eight roundings an entry, here and in the reference, so 2^-49."""
    rng = np.random.default_rng(K)
    n = rng.integers(1, K, D)
    n[::3] = 0
    diag = rng.uniform(1.0, 2.0, (D, K))
    diag[1::3] *= 2.0 ** 32
    err, kappa = _draw(K, 1.0, n, prec, (rng.standard_normal((D, K)), diag[:, :, None] * np.eye(K)))
    own = np.arange(D) % 3 < 2
    assert (err[own] <= 2.0 ** -49).all(), np.sort(err[own])[-5:] * 2.0 ** 49
    assert (err[~own] <= 4 * K * 2.0 ** -44 * kappa[~own]).all()


@pytest.mark.parametrize("K", [16, 24])
def test_low_noise_rows_stay_near_the_speed_of_the_others(K):
    """K / 2 observations a row: at sigma = 2e-3 nearly every row loses its pivots' bits, at 0.5 none.
    Drawn by a lane each, such rows made the sweep 7 times as long."""
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(K)
    N, n, Dc = 60_000, K // 2, 20_000
    row = np.repeat(np.arange(N), n)
    col = (rng.integers(0, Dc, N)[:, None] + np.arange(n) * 97).reshape(-1) % Dc
    X, W = rng.standard_normal((N, K)), rng.standard_normal((Dc, K))
    best = {}
    for sigma in (0.5, 3e-3 if K == 24 else 2e-3):
        y = (X[row] * W[col]).sum(1) + sigma * rng.standard_normal(len(row))
        m = bmf.BMF(N, Dc, row, col, y, K, sigma ** -2, "fp32", X0=X, W0=W, seed=1)
        m.sweep(0, 3, None)
        best[sigma] = np.inf
        for _ in range(4):
            t = time.perf_counter()
            m.sweep(0, 10, None)
            best[sigma] = min(best[sigma], time.perf_counter() - t)
        m.close()
    a, b = best.values()
    assert b < 4 * a, (a, b)
