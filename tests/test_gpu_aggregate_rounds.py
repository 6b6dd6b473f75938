"""bmf_aggregate_static in several rounds: more rows than one round's scratch holds, more submodels
than one row's pairs fit, and odd sizes at the edges of a block, against Eq. 14 / Algorithm 2.

Tolerance: Lambda* and its right-hand side are sums of J terms accumulated in FP64, relative
error at most about 2 J 2^-53 (5e-10 at the largest J here) of the sum of the terms' magnitudes,
which is about 12 times the result; K = 1 solves by one division.  The K > 1 cases follow the
1e-9 of the aggregation's other tests."""
import numpy as np
import pytest

import oracle
from pairing import assert_rows_close

pytestmark = pytest.mark.gpu


def _call(mu, lam):
    import torch
    from paper_1703_00734_gb300 import bmf
    J, R, K = mu.shape
    dm, dl = torch.from_numpy(mu).cuda(), torch.from_numpy(lam).cuda()
    out = torch.full((R, K), float("nan"), dtype=torch.float64, device="cuda")
    n = bmf.aggregate_static(K, R, J, dm.data_ptr(), dl.data_ptr(), out.data_ptr(), 1e-6,
                             torch.cuda.current_stream().cuda_stream)
    return out.cpu().numpy(), n


@pytest.mark.parametrize("R,J", [(1_500_000, 2), (2, 2_100_000)])
def test_rounds_of_rows_and_of_submodels(R, J):
    rng = np.random.default_rng(R)
    mu = rng.standard_normal((J, R, 1))
    lam = rng.uniform(1.0, 2.0, (J, R, 1, 1))
    lam[0] = 1.5
    got, n = _call(mu, lam)
    l, m = lam[:, :, 0, 0], mu[:, :, 0]
    dif = l[1:] - l[0]
    bad = ~(dif > 0)
    eps = 1e-6 * np.maximum(1.0, l[0])
    lj = np.where(bad, dif + np.abs(dif) + eps + l[0], l[1:])
    want = ((2.0 - J) * l[0] * m[0] + (lj * m[1:]).sum(0)) / ((2.0 - J) * l[0] + lj.sum(0))
    assert n == int(bad.sum())
    np.testing.assert_allclose(got[:, 0], want, rtol=1e-8, atol=1e-9)


@pytest.mark.parametrize("K,R,J", [(2, 1, 2), (7, 31, 3), (13, 33, 5), (16, 97, 2)])
def test_odd_sizes_match_the_oracle(K, R, J):
    rng = np.random.default_rng(K)
    A = rng.standard_normal((J, R, K, K))
    lam = A @ A.transpose(0, 1, 3, 2) / K + np.eye(K)
    mu = rng.standard_normal((J, R, K))
    # keep the aggregated precision definite: the correction makes every difference so
    want, _, nc = oracle.aggregate(mu, lam, 1e-6)
    got, n = _call(mu, lam)
    assert n == nc
    assert_rows_close(got, want, 1e-9, f"K={K}")
