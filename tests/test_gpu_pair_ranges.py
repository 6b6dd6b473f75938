"""Rows whose terms are inside a float pair's range but whose right-hand side or solution leaves FP32's
exponents: the draw of the reduced-precision modes is FP64's, finite and as exact as its Gram sums.

Both factors carry per-row priors.  X is pinned to its prior means by a precision of 1e60, so the
W draw that ends the sweep has G = sum x x^T and r = sum y x of known x.  Tolerance: x rounded to
FP32 and FP32 sums of n terms leave (n + 3) 2^-24 of G and of r's terms, at most 1e-5 here, and the
precisions have condition numbers below 10."""
import numpy as np
import pytest

from paper_1703_00734_gb300 import synth

pytestmark = pytest.mark.gpu
N, D = 40, 20


def _sweep(K, tau, val, x_scale, muW, LamW, prec="fp32"):
    """W after one sweep and the same by FP64 arithmetic."""
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(K)
    row, col = np.repeat(np.arange(N), D), np.tile(np.arange(D), N)
    keep = rng.random(N * D) < 0.6
    row, col = row[keep], col[keep]
    y = val * rng.uniform(0.5, 1.0, len(row))
    muX = x_scale * rng.standard_normal((N, K))
    m = bmf.BMF(N, D, row, col, y, K, tau, prec, order="none", center=False,
                X0=muX, W0=0.1 * rng.standard_normal((D, K)))
    m.set_prior(0, bmf.FACTOR_X, muX, np.broadcast_to(1e60 * np.eye(K), (N, K, K)).copy())
    m.set_prior(0, bmf.FACTOR_W, np.broadcast_to(muW, (D, K)).copy(), np.broadcast_to(LamW, (D, K, K)).copy())
    dr = synth.sweep_draws([(N, D)], K, float(K), synth.rng_for(0, 1))
    m.sweep(0, 1, dr)
    X, W, _ = m.get_state(0)
    m.close()
    z = dr[-D * K:].reshape(D, K)
    want = np.empty((D, K))
    for j in range(D):
        x = X[row[col == j]]
        L = np.linalg.cholesky(LamW + tau * x.T @ x)
        b = LamW @ muW + tau * x.T @ y[col == j]
        want[j] = np.linalg.solve(L.T, np.linalg.solve(L, b) + z[j])
    return W, want


def _check(W, want):
    err = np.linalg.norm(W - want, axis=1) / np.linalg.norm(want, axis=1)
    assert np.isfinite(W).all() and err.max() < 1e-3, err


@pytest.mark.parametrize("K", [9, 10, 16, 20, 40])
def test_a_product_beyond_fp32(K):
    """tau = 2^60 and r about 2^68, each a pair's: tau r is not."""
    W, want = _sweep(K, 2.0 ** 60, 2.0 ** 66.5, 1.0, np.zeros(K), 2.0 ** 60 * 20.0 * np.eye(K))
    assert np.abs(want).max() > 2.0 ** 58
    _check(W, want)


@pytest.mark.parametrize("K", [9, 10, 16, 20, 40])
def test_a_solution_beyond_fp32(K):
    """A prior precision of 2^-59.5 with a mean of 2^129.4: their product is a pair's, the draw is not."""
    W, want = _sweep(K, 2.0 ** -59.5, 1.0, 0.05, np.full(K, 2.0 ** 129.4), 2.0 ** -59.5 * np.eye(K))
    assert np.abs(want).max() > 2.0 ** 128
    _check(W, want)


@pytest.mark.parametrize("K", [10, 16, 20, 40])
def test_ordinary_scales(K):
    W, want = _sweep(K, 4.0, 1.0, 1.0, np.ones(K), 4.0 * np.eye(K), "bf16" if K == 16 else "fp32")
    err = np.linalg.norm(W - want, axis=1) / np.linalg.norm(want, axis=1)
    assert err.max() < (0.1 if K == 16 else 1e-4), err
