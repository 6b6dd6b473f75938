"""The team conditional at the edges of its layout: matrices below, at and above a team's batch of
entries, the largest K, every number of lanes that fits (bit-identical among themselves), rows with a
sum over several work items and rows without observations.  Tolerance: one transition in FP64, as
everywhere against the oracle (1e-9 per row)."""
import numpy as np
import pytest

from paper_1703_00734_gb300 import synth
from pairing import Pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,lanes", [(13, (2, 4, 8, 16, 32)), (17, (2, 4, 8, 16, 32)), (33, (4, 8, 16, 32)),
                                     (40, (4, 8, 16, 32)), (63, (16, 32)), (64, (16, 32))])
def test_team_conditional(K, lanes):
    d = synth.make_workload(None, N=131, D=1100, M=9000, pattern="zipf", K=K, sigma=0.5, tau=4.0, seed=80 + K,
                            s_row=1.2, s_col=1.2)
    keep = d["row"] != 7
    for k in ("row", "col", "val"):
        d[k] = d[k][keep]
    first = None
    for n in lanes:
        pr = Pair(d, K)
        pr.m.set_schedule(1, 1, 4, 0.0, 0, n)
        assert pr.m.get_schedule()["cond_lanes"] == n
        pr.run_stage(1, 1)
        if first is None:
            pr.compare_subset(0)
            first = pr.m.get_state(0)
        for a, b in zip(first[:2], pr.m.get_state(0)[:2]):
            np.testing.assert_array_equal(a, b)
        pr.m.close()
