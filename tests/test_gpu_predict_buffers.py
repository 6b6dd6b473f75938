"""Predictions before and after the device generator's tables grow: the prediction buffer is its own."""
import numpy as np
import pytest

from paper_1703_00734_gb300 import synth

pytestmark = pytest.mark.gpu


def test_generator_tables_do_not_take_the_prediction_buffer():
    from paper_1703_00734_gb300 import bmf
    K = 4
    d = synth.make_workload(None, N=60, D=40, M=900, pattern="uniform", K=K, sigma=0.5, tau=4.0, seed=3, s_row=1.2,
                            s_col=1.2)
    m = bmf.BMF(d["N"], d["D"], d["row"], d["col"], d["val"], K, d["tau"], "fp64", X0=d["X0"], W0=d["W0"], seed=1)
    T = K + 3
    dr = np.concatenate([synth.sweep_draws([(d["N"], d["D"])], K, float(K), synth.rng_for(1, t)) for t in range(T)])
    m.stage(1, T, dr)                               # host draws: the generator has no tables yet
    row, col = np.arange(60, dtype=np.int32), np.arange(60, dtype=np.int32) % 40
    first, _ = m.predict(row, col)
    m.generate_draws(1)                             # ... now it has
    second, _ = m.predict(row, col)
    m.close()
    np.testing.assert_array_equal(first, second)
