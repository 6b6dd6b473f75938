"""lambda-means where its two forms meet: rows that open more clusters than the fast form keeps (32),
up to one per sample, among rows that open few; samples that lie exactly on lambda or half way
between centres, where the FP32 distances cannot decide; NaN and infinite samples.  Assignments
bit-identical to the oracle's; fits at the 1e-9 of the other summary tests."""
import numpy as np
import pytest

import oracle
from pairing import assert_rows_close

pytestmark = pytest.mark.gpu


def _fit(x, lam, C=3, mode="gmm"):
    import torch
    from paper_1703_00734_gb300 import bmf
    return {k: v.cpu().numpy() for k, v in bmf.fit_summaries(torch.from_numpy(x).cuda(), mode, lam, C=C).items()}


@pytest.mark.parametrize("S,K", [(8, 1), (31, 2), (33, 3), (100, 5), (256, 32)])
def test_many_clusters_and_exact_ties(S, K):
    rng = np.random.default_rng(S)
    x = rng.standard_normal((S, 40, K)) * 0.05
    x[:, 1::4] += 10.0 * np.arange(S)[:, None, None]              # a cluster per sample
    x[:, 2::4] = rng.integers(0, 3, (S, 10, K))                    # lattice: ties and exact lambda
    x[:, 3::4] += 4.0 * (np.arange(S)[:, None, None] % min(S, 40))  # about 40 clusters
    lam = 1.0
    got = _fit(x, lam) if S >= K + 1 and K < 8 else None
    for r in range(40):
        a, _ = oracle.lambda_means(np.ascontiguousarray(x[:, r]), lam)
        if got is None:
            break
        np.testing.assert_array_equal(got["assign"][r], a, err_msg=f"row {r}")
    y = np.ascontiguousarray(x[:, 0::4])                           # ordinary rows keep their fits
    if S >= K + 1:
        g, w = _fit(y, lam), oracle.fit_summaries(y, "gmm", lam=lam, C=3)
        assert_rows_close(g["pooled_Lam"].reshape(10, -1), w["pooled_Lam"].reshape(10, -1), 1e-9, "pooled")
        np.testing.assert_array_equal(g["pi"], w["pi"])


def test_a_dropped_component_and_a_row_without_one():
    """The largest cluster repeats one point (singular): it is dropped and the next one leads; a row
    whose clusters are all too small takes all its samples."""
    rng = np.random.default_rng(0)
    K, S = 3, 60
    x = rng.standard_normal((S, 3, K)) * 0.1
    x[:35, 0] = 5.0
    x[:, 1] += 9.0 * (np.arange(S)[:, None] // 3)
    g, w = _fit(x, 2.0), oracle.fit_summaries(x, "gmm", lam=2.0, C=3)
    np.testing.assert_array_equal(g["pi"], w["pi"])
    assert_rows_close(g["mu"].reshape(9, K), w["mu"].reshape(9, K), 1e-9, "mu")
    assert_rows_close(g["pooled_Lam"].reshape(3, -1), w["pooled_Lam"].reshape(3, -1), 1e-9, "pooled")


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_samples(bad):
    """A non-finite sample is nearest to nothing and ends in a cluster of its own, as in the oracle;
    with all samples in one Gaussian its covariance is not positive definite."""
    from paper_1703_00734_gb300 import bmf
    x = np.random.default_rng(1).standard_normal((20, 4, 3))
    x[7, 2, 1] = bad
    g = _fit(x, 1e3)
    for r in range(4):
        np.testing.assert_array_equal(g["assign"][r], oracle.lambda_means(np.ascontiguousarray(x[:, r]), 1e3)[0])
    with pytest.raises(bmf.BmfError) as e:
        _fit(x, 1e3, C=1, mode="mm")
    assert e.value.status == 3
