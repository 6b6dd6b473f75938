"""Rows that open more clusters than the first launch of the summaries keeps: assignments equal to the
oracle's, element by element, in both forms of the second launch (FP32 distances where 2 S centres
fit beside the samples, FP64 where they do not: S = 1024, K = 8), up to a cluster per sample at the
largest S K, and their cost."""
import time

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,K", [(33, 1), (200, 10), (256, 32), (512, 16), (1024, 8)])
@pytest.mark.parametrize("mode", ["dm", "gmm"])
def test_assignments(S, K, mode):
    import torch
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(S + K)
    R = 16
    x = rng.standard_normal((S, R, K)) * 0.05
    x[:, 1::4] += 10.0 * np.arange(S)[:, None, None]                  # a cluster per sample
    x[:, 2::4] = rng.integers(0, 3, (S, R // 4, K))                   # lattice: ties and exact lambda
    x[:, 3::4] += 4.0 * (np.arange(S)[:, None, None] % min(S, 40))    # about 40 clusters
    got = bmf.fit_summaries(torch.from_numpy(x).cuda(), mode, 1.0, C=1 if mode == "dm" else 3)["assign"].cpu().numpy()
    for r in range(R):
        want, _ = oracle.lambda_means(np.ascontiguousarray(x[:, r]), 1.0)
        np.testing.assert_array_equal(got[r], want, err_msg=f"row {r}")


def test_many_clusters_cost_what_their_distances_do():
    """60 clusters need 60 times the distances of one, in a pass of about the same work per cluster
    otherwise: 8 times the call (60 times when the rows shared two warps per SM in FP64)."""
    import torch
    from paper_1703_00734_gb300 import bmf
    g = torch.Generator(device="cuda").manual_seed(1)
    few = 0.05 * torch.randn(200, 20_000, 10, generator=g, device="cuda", dtype=torch.float64)
    many = few + 4.0 * (torch.arange(200, device="cuda") % 60)[:, None, None]

    def best(x, lam):
        out = np.inf
        for _ in range(4):
            torch.cuda.synchronize()
            t = time.perf_counter()
            bmf.fit_summaries(x, "gmm", lam, 3)
            out = min(out, time.perf_counter() - t)
        return out

    a, b = best(few, 1e9), best(many, 1.0)
    assert b < 25 * a, (a, b)
