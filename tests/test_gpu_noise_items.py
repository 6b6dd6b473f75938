"""Sampled noise precisions where a column's squared residuals come from several work items (1,024
entries each): columns of 1,024 entries and one more, of 3 items, of all rows, and empty ones.
Tolerance: three sweeps in FP64 against the oracle (1e-8 per row)."""
import numpy as np
import pytest

import oracle
from pairing import assert_rows_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["column", "global"])
@pytest.mark.parametrize("K", [3, 4, 20])
def test_columns_of_several_items(K, mode):
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(K)
    N, D, T, seed = 4200, 30, 3, 31
    count = np.r_[1024, 1025, 2049, 3000, N, 0, rng.integers(1, 300, D - 6)]
    col = np.repeat(np.arange(D), count)
    row = np.concatenate([rng.choice(N, k, replace=False) for k in count])
    X0, W0 = 0.5 * rng.standard_normal((N, K)), 0.5 * rng.standard_normal((D, K))
    val = rng.standard_normal(len(row)) * (0.3 + 0.1 * (col % 7))
    m = bmf.BMF(N, D, row, col, val, K, 2.0, "fp64", X0=X0, W0=W0, seed=seed, noise=mode, noise_a0=2.0, noise_b0=0.5)
    p = oracle.plan(N, D, row, col, val, 1, 1)
    noise = oracle.NoiseModel(mode, 2.0, 0.5, 2.0)
    chains = oracle.setup_stage_chains(p, 1, X0[p.row_perm], W0[p.col_perm], K, {})
    oracle.run_stage(p, 1, chains, K, 2.0, oracle.NWPrior(K),
                     lambda t: oracle.gen_batch_draws(p.stage_subsets(1), K, float(K), seed, t + 1, noise), T, 0, 1, noise)
    m.stage(1, T, None)
    X, W, _ = m.get_state(0)
    tau, st = m.get_noise(0), chains[0]
    m.close()
    assert_rows_close(tau[:, None], st.tau_col[:, None], 1e-8, "tau")
    assert_rows_close(X, st.X, 1e-8, "X")
    assert_rows_close(W, st.W, 1e-8, "W")
