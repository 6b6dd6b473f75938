"""The conditional draw of the reduced-precision modes: float pairs at 9 <= K <= 48, FP64 around
them, and the FP64 fallback for rows outside a pair's range.

Rows without observations have zero Gram sums, so their draw is x = mu + L^{-T} z with the row's
own prior, and its only error is the factorisation's.  Tolerance: a pair operation is off by at
most 2^-44, each entry takes at most K of them, so the backward error of the factor is below
K 2^-44 and |dx| below 4 K 2^-44 cond(Lambda) |x| (the FP64 rows, whose reduced-precision pivot
is off by 2^-41 at most, below 4 K 2^-41 cond(Lambda) |x|)."""
import numpy as np
import pytest

from paper_1703_00734_gb300 import synth

pytestmark = pytest.mark.gpu

ROWS = 70          # a full conditional block and a partial one


def _model(K, prec, seed=0):
    """A matrix whose rows from 8 on have no observations, its draws of one sweep and the z of X."""
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(seed)
    row, col = np.repeat(np.arange(8), 6), np.tile(np.arange(6), 8)
    m = bmf.BMF(ROWS, 6, row, col, rng.standard_normal(48), K, 4.0, prec, order="none",
                X0=0.1 * rng.standard_normal((ROWS, K)), W0=0.1 * rng.standard_normal((6, K)))
    dr = synth.sweep_draws([(ROWS, 6)], K, float(K), synth.rng_for(seed, 1))
    H = 2 * (K + K * (K - 1) // 2 + K)
    return m, dr, dr[H:H + ROWS * K].reshape(ROWS, K)


def _priors(K, rng, cond=30.0):
    A = np.linalg.qr(rng.standard_normal((ROWS, K, K)))[0]
    ev = np.exp(rng.uniform(0.0, np.log(cond), (ROWS, K)))
    Lam = (A * ev[:, None, :]) @ A.transpose(0, 2, 1)
    return rng.standard_normal((ROWS, K)), 0.5 * (Lam + Lam.transpose(0, 2, 1))


def _want(mu, Lam, z):
    L = np.linalg.cholesky(Lam)
    return mu + np.stack([np.linalg.solve(L[r].T, z[r]) for r in range(len(mu))])


@pytest.mark.parametrize("K", [1, 8, 9, 12, 13, 16, 17, 24, 25, 32, 33, 48, 49, 64])
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_rows_without_observations_follow_their_priors(K, prec):
    m, dr, z = _model(K, prec)
    mu, Lam = _priors(K, np.random.default_rng(K))
    m.set_prior(0, 0, mu, Lam)
    m.sweep(0, 1, dr)
    X, _, _ = m.get_state(0)
    m.close()
    want = _want(mu, Lam, z)[8:]
    unit = 2.0 ** (-44 if 9 <= K <= 48 else -41)
    err = np.linalg.norm(X[8:] - want, axis=1) / np.linalg.norm(want, axis=1)
    assert err.max() <= 4 * K * unit * 30.0, err.max()


@pytest.mark.parametrize("K", [10, 16, 20, 40])
def test_rows_outside_a_pairs_range_are_drawn_in_fp64(K):
    """Scales far beyond FP32's exponents, and conditioning beyond a pair's 48 bits, row by row
    among ordinary rows: the draw keeps FP64's accuracy relative to each row's own scale."""
    m, dr, z = _model(K, "fp32", 1)
    mu, Lam = _priors(K, np.random.default_rng(K))
    scale = np.ones(ROWS)
    scale[10::9] = 1e60          # precision 1e60: draws of 1e-30
    scale[11::9] = 1e-60
    scale[12::9] = 1e22          # beyond 2^70, within FP32's exponents
    Lam = Lam * scale[:, None, None]
    mu = mu / np.sqrt(scale)[:, None]
    near = np.arange(13, ROWS, 9)          # lambda_max / lambda_min = 1e13
    A = np.linalg.qr(np.random.default_rng(7).standard_normal((len(near), K, K)))[0]
    ev = np.ones((len(near), K))
    ev[:, 0] = 1e-13
    Lam[near] = (A * ev[:, None, :]) @ A.transpose(0, 2, 1)
    Lam[near] = 0.5 * (Lam[near] + Lam[near].transpose(0, 2, 1))
    m.set_prior(0, 0, mu, Lam)
    m.sweep(0, 1, dr)
    X, _, _ = m.get_state(0)
    m.close()
    want = _want(mu, Lam, z)
    err = np.linalg.norm(X - want, axis=1) / np.linalg.norm(want, axis=1)
    plain = np.setdiff1d(np.arange(8, ROWS), near)
    assert err[plain].max() <= 4 * K * 2.0 ** -41 * 30.0, err[plain].max()
    # FP64 itself leaves K 2^-52 cond = 1e13 K 2^-52 of these
    assert err[near].max() <= 16 * K * 2.0 ** -52 * 1e13, err[near].max()


@pytest.mark.parametrize("K", [10, 16, 20, 40])
def test_an_indefinite_row_is_reported(K):
    from paper_1703_00734_gb300 import bmf
    m, dr, _ = _model(K, "fp32", 2)
    mu, Lam = _priors(K, np.random.default_rng(K))
    Lam[37, K - 1, K - 1] = -1.0
    m.set_prior(0, 0, mu, Lam)
    with pytest.raises(bmf.BmfError) as e:
        m.sweep(0, 1, dr)
    assert e.value.status == 3
    m.close()
