"""The adjoint where a row's data term comes from several work items (1,024 observations each: 3, 5 and
7 items, so that the rows' pass meets every remainder of its four items in flight), and where its
blocks step through the rows more than once, with a last warp that is not full.

Tolerance per entry, from the operations in FP32 (u = 2^-24): a residual is off by (K + 2) u times the
magnitudes it sums, a gradient entry by that times |partner| and by the additions of its terms (at
most 300 in a row: 256 of a lane, the reductions and the items), the prior term by (2 K + 4) u of its
magnitudes; the values alike.  The oracle is FP64."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
U, DEPTH = 2.0 ** -24, 300


def _check(N, D, row, col, K, seed):
    import torch
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(seed)
    X, W = (rng.standard_normal((n, K)).astype(np.float32) for n in (N, D))
    y = rng.standard_normal(len(row)) + (X[row].astype(np.float64) * W[col]).sum(1)
    y = y.astype(np.float32).astype(np.float64)
    m = bmf.BMF(N, D, row, col, y, K, 4.0, "fp32", order="none", center=False)

    def prior():
        A = rng.standard_normal((K, K)) * 0.3
        return rng.standard_normal(K), A @ A.T + np.eye(K)
    (mX, LX), (mW, LW) = prior(), prior()
    for f, n, mu, L in ((bmf.FACTOR_X, N, mX, LX), (bmf.FACTOR_W, D, mW, LW)):
        m.set_prior(0, f, np.tile(mu, (n, 1)), np.tile(L, (n, 1, 1)))
    ld, la = (K + 3) // 4 * 4, np.log(4.0)
    dev = [torch.zeros((len(A), ld), dtype=torch.float32, device="cuda") for A in (X, W)]
    for t, A in zip(dev, (X, W)):
        t[:, :K] = torch.from_numpy(A).cuda()
    gX, gW = (torch.full_like(t, 7.0) for t in dev)
    v, ga = m.logjoint_grad(0, dev[0].data_ptr(), dev[1].data_ptr(), ld, la, gX.data_ptr(), gW.data_ptr())
    m.close()
    X64, W64 = X.astype(np.float64), W.astype(np.float64)
    o = np.lexsort((col, row))
    row, col, y = row[o].astype(np.int32), col[o].astype(np.int32), y[o]
    wX, wW, wa, wv = oracle.logjoint_grad(row, col, y, X64, W64, la, mX, LX, mW, LW)
    r = y - (X64[row] * W64[col]).sum(1)
    er = (K + 2) * U * (np.abs(y) + (np.abs(X64[row]) * np.abs(W64[col])).sum(1))   # of a residual
    bv = 0.0
    for own, part, F, P, mu, L, g, want in ((row, col, X64, W64, mX, LX, gX, wX), (col, row, W64, X64, mW, LW, gW, wW)):
        tol = np.zeros_like(F)
        np.add.at(tol, own, 4.0 * (er + DEPTH * U * np.abs(r))[:, None] * np.abs(P[part]))
        pm = np.abs(F) @ np.abs(L).T + np.abs(L @ mu)
        tol += (2 * K + 4) * U * pm + 4 * U * np.abs(want)
        g = g.cpu().numpy()
        assert (np.abs(g[:, :K] - want) <= tol).all(), (np.abs(g[:, :K] - want) / tol).max()
        assert (g[:, K:] == 0).all()
        bv += (2 * K + 4) * U * (np.abs(F) * (pm + 2 * np.abs(L @ mu))).sum()
        wv += 0.5 * len(F) * mu @ L @ mu            # the value drops the constant of the priors
    br = 4.0 * (2 * np.abs(r) * er + DEPTH * U * r * r).sum()
    assert abs(v - wv) <= 0.5 * (br + bv) + 1e-12 * abs(wv), (v, wv, br, bv)
    assert abs(ga - wa) <= 0.5 * br + 1e-12 * abs(wa)


@pytest.mark.parametrize("K", [5, 16, 20, 64])
def test_rows_of_several_items(K):
    n = 7200
    heavy = (2500, 4097, 7168)                       # 3, 5 and 7 items
    pairs = {(q, c) for q, k in enumerate(heavy) for c in range(n - k, n)}
    pairs |= {(c, q) for q, k in enumerate(heavy) for c in range(n - k, n)}
    row, col = np.array(sorted(pairs)).T
    _check(n, n, row, col, K, K)


@pytest.mark.parametrize("K,N,D", [(5, 40_003, 39_001), (64, 25_003, 19_457)])
def test_more_rows_than_the_blocks_take_at_once(K, N, D):
    rng = np.random.default_rng(K)
    key = np.unique(rng.integers(0, N * D, 60_000))
    _check(N, D, key // D, key % D, K, K)
