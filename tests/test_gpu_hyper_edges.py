"""The hyperparameter draw on either side of its rules: the short chain up to K = 16 and the plain one
above, and there factor blocks of 64 statistics chunks of 64 rows, summed by the draw itself, and of
65.  Tolerance: one transition in FP64 (1e-9 per row)."""
import pytest

from paper_1703_00734_gb300 import synth
from pairing import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [15, 16, 17])
@pytest.mark.parametrize("N,D", [(4096, 65), (4097, 64), (63, 4097)])
def test_hyperparameter_draw(K, N, D):
    d = synth.make_workload(None, N=N, D=D, M=20 * max(N, D), pattern="uniform", K=K, sigma=0.5, tau=4.0, seed=60 + K,
                            s_row=1.2, s_col=1.2)
    pr = Pair(d, K)
    pr.run_stage(1, 1)
    pr.compare_subset(0)
