"""Several Langevin moves in one call: unadjusted steps, which follow one another in place, and
Metropolis-adjusted ones, whose second step starts from the gradients that the first one's decision
left (kept or taken over).

Tolerance: one step agrees to 1e-5 per row (as everywhere against the FP64 oracle) and later steps
multiply what is off by 1 + (eps / 2) |H|, H bounded by the largest sum of squares of a row's
partners, its cross terms and its prior."""
import numpy as np
import pytest

import oracle
from test_gpu_adjoint import _close_rows, _dev, _oracle_grad, _setup

pytestmark = pytest.mark.gpu
K, LA = 6, np.log(1 / 0.09)


def _step(s, X, W, prior, eps, xi):
    gX, gW, _, v = _oracle_grad(s, X, W, LA, prior)
    Xn = X + 0.5 * eps * gX + np.sqrt(eps) * xi[:s.n * K].reshape(s.n, K)
    Wn = W + 0.5 * eps * gW + np.sqrt(eps) * xi[s.n * K:].reshape(s.d, K)
    return gX, gW, v, Xn, Wn


def _towards_the_mode(s, X, W, prior):
    X, W = X.astype(np.float64), W.astype(np.float64)
    for _ in range(400):
        gX, gW, *_ = _oracle_grad(s, X, W, LA, prior)
        X, W = X + 2e-4 * gX, W + 2e-4 * gW
    return X.astype(np.float32), W.astype(np.float32)


def _growth(s, X, W, prior, eps):
    row = np.repeat(np.arange(s.n), np.diff(s.rptr))
    x2, w2 = (X ** 2).sum(1), (W ** 2).sum(1)
    hx, hw = np.bincount(row, w2[s.ridx], s.n).max(), np.bincount(s.ridx, x2[row], s.d).max()
    L = max(np.abs(prior["LamXr"]).sum(2).max(), np.abs(prior["LamWr"]).sum(2).max())
    return 1 + 0.5 * eps * (np.exp(LA) * 2 * max(hx, hw) + L)


def test_unadjusted_steps_in_place():
    torch, _, m, s, X, W, ld, prior = _setup(K, False)
    eps, n = 1e-4, 3
    xi = np.random.default_rng(8).standard_normal((n, (s.n + s.d) * K)).astype(np.float32)
    dX, dW = _dev(torch, X, ld), _dev(torch, W, ld)
    dX[:, K:], dW[:, K:] = 3.0, 5.0                       # padding is the caller's
    acc, value = m.langevin(0, n, dX.data_ptr(), dW.data_ptr(), ld, LA, eps, torch.from_numpy(xi).cuda().data_ptr())
    assert acc == n
    g, tol, Xc, Wc = _growth(s, X, W, prior, eps), 0.0, X, W
    for q in range(n):
        tol = tol * g + 1e-5
        *_, Xc, Wc = _step(s, Xc, Wc, prior, eps, xi[q])
    _close_rows(dX.cpu().numpy()[:, :K], Xc, tol, "X")
    _close_rows(dW.cpu().numpy()[:, :K], Wc, tol, "W")
    assert (dX[:, K:] == 3.0).all() and (dW[:, K:] == 5.0).all()
    # the value is the final state's
    h = [torch.empty_like(dX), torch.empty_like(dW)]
    v, _ = m.logjoint_grad(0, dX.data_ptr(), dW.data_ptr(), ld, LA, h[0].data_ptr(), h[1].data_ptr())
    assert v == value
    m.close()


@pytest.mark.parametrize("decide", [(1, 1), (1, 0), (0, 1), (0, 0), (1, 0, 1)])
def test_adjusted_steps_follow_the_decisions(decide):
    torch, _, m, s, X, W, ld, prior = _setup(K, False)
    X, W = _towards_the_mode(s, X, W, prior)              # where a log-ratio is about -10
    eps = 5e-4
    xi = np.random.default_rng(9).standard_normal((len(decide), (s.n + s.d) * K)).astype(np.float32)
    g, tol, Xc, Wc, us = _growth(s, X, W, prior, eps), 0.0, X.astype(np.float64), W.astype(np.float64), []
    for q, take in enumerate(decide):
        gX, gW, v, Xn, Wn = _step(s, Xc, Wc, prior, eps, xi[q])
        pX, pW, vn, _, _ = _step(s, Xn, Wn, prior, eps, xi[q])
        back = ((Xc - Xn - 0.5 * eps * pX) ** 2).sum() + ((Wc - Wn - 0.5 * eps * pW) ** 2).sum()
        fwd = ((Xn - Xc - 0.5 * eps * gX) ** 2).sum() + ((Wn - Wc - 0.5 * eps * gW) ** 2).sum()
        logA = vn - v + (fwd - back) / (2 * eps)
        assert -300 < logA < -4, logA                     # both decisions have room for a margin of 3
        us.append(np.exp(logA - 3.0 if take else logA + 3.0))
        if take:
            Xc, Wc, tol = Xn, Wn, tol * g + 1e-5
    dX, dW = _dev(torch, X, ld), _dev(torch, W, ld)
    acc, _ = m.langevin(0, len(decide), dX.data_ptr(), dW.data_ptr(), ld, LA, eps,
                        torch.from_numpy(xi).cuda().data_ptr(), uniforms=us)
    assert acc == sum(decide)
    _close_rows(dX.cpu().numpy()[:, :K], Xc, max(tol, 1e-12), "X")
    _close_rows(dW.cpu().numpy()[:, :K], Wc, max(tol, 1e-12), "W")
    m.close()
