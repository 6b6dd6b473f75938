"""A kernel's limit of dynamic shared memory belongs to the kernel, not to a context or a launch: every
launch sets the same one (common.cuh), or two host threads could take each other's away between
setting it and launching."""
import os
import threading

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_00734_gb300", "csrc")


def test_one_place_sets_the_limit():
    where = [f for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh", ".h", ".cpp"))
             and "MaxDynamicSharedMemorySize" in open(os.path.join(CSRC, f)).read()]
    assert where == ["common.cuh"]


@pytest.mark.gpu
def test_two_contexts_on_two_threads():
    """Sides whose launches of one kernel take 190 and 95 KB (9,000 and 19,000 rows at K = 32), two
    chains of one seed at the same time: no call fails and both give the lone chain's states."""
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(0)
    N, D, K = 9_000, 19_000, 32
    cell = np.unique(rng.integers(0, N * D, 300_000))
    row, col = cell // D, cell % D
    y = rng.standard_normal(len(cell))
    out = {}

    def chain(name):
        m = bmf.BMF(N, D, row, col, y, K, 4.0, "fp32", X0=x0, W0=w0, seed=1)
        for _ in range(20):
            m.sweep(0, 5, None)
        out[name] = m.get_state(0)[:2]
        m.close()

    x0, w0 = 0.1 * rng.standard_normal((N, K)), 0.1 * rng.standard_normal((D, K))
    chain("alone")
    pair = [threading.Thread(target=chain, args=(k,)) for k in range(2)]
    for t in pair:
        t.start()
    for t in pair:
        t.join()
    for k in range(2):
        for a, b in zip(out["alone"], out[k]):
            np.testing.assert_array_equal(a, b)
