"""The hyperparameter draw at the edges of its rules: the short chain (K <= 16) and the plain one, and factor blocks of up to 64 statistics
chunks of 64 rows, summed by the draw itself, against longer ones.  Tolerance: one transition in
FP64, as everywhere against the oracle (1e-9 per row)."""
import pytest

from paper_1703_00734_gb300 import synth
from pairing import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,N,D", [(1, 65, 2), (2, 4096, 33), (3, 4097, 64), (31, 300, 40), (32, 90, 4097),
                                   (33, 129, 64), (48, 4096, 70), (49, 200, 60)])
def test_hyperparameter_draw(K, N, D):
    d = synth.make_workload(None, N=N, D=D, M=min(20 * max(N, D), N * D // 2), pattern="uniform", K=K, sigma=0.5,
                            tau=4.0, seed=60 + K, s_row=1.2, s_col=1.2)
    pr = Pair(d, K)
    pr.run_stage(1, 1)
    pr.compare_subset(0)
