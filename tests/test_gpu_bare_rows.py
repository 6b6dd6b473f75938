"""Rows without observations whose prior is their own, which the reduced-precision modes draw apart from
the others (9 <= K <= 16), from factors that one call's sweeps share: the sweeps of one call and calls
of one sweep give the same bits, under every schedule, with their moments; a mixture prior's component
changes between the sweeps of a call; a prior that is not positive definite is refused.  (How exact the
draws are: test_gpu_pair_rows.py.)"""
import numpy as np
import pytest

from paper_1703_00734_gb300 import synth

pytestmark = pytest.mark.gpu
N, D = 300, 131


def _context(K, prec, sched, bad=None):
    from paper_1703_00734_gb300 import bmf
    rng = np.random.default_rng(K)
    key = rng.choice(N * D, 250, replace=False)          # about 130 of 300 and 20 of 131 rows have none
    row, col = key // D, key % D
    m = bmf.BMF(N, D, row, col, rng.standard_normal(len(key)), K, 4.0, prec, order="none", seed=7, moments="full")
    m.set_schedule(*sched)
    for f, n in ((bmf.FACTOR_X, N), (bmf.FACTOR_W, D)):
        A = rng.standard_normal((n, K, 2 * K))
        Lam = A @ A.transpose(0, 2, 1)
        if f == bmf.FACTOR_X and bad is not None:
            empty = np.setdiff1d(np.arange(N), row)
            bad = empty[bad]
            Lam[bad, -1, -1] = -1.0
        m.set_prior(0, f, rng.standard_normal((n, K)), Lam)
    return m, bad


@pytest.mark.parametrize("K,prec", [(9, "fp32"), (12, "bf16"), (13, "tf32"), (16, "fp32")])
def test_one_call_equals_calls_of_one_sweep(K, prec):
    from paper_1703_00734_gb300 import bmf
    a, _ = _context(K, prec, (1, 1, 4, 0.0, 0, 0))
    S1 = S2 = 0.0
    for _ in range(3):
        a.sweep(0, 1, None)
        X, W, _ = a.get_state(0)
        S1, S2 = S1 + X, S2 + np.einsum("ni,nj->nij", X, X)
    mom = [a.get_moments(0, f) for f in (bmf.FACTOR_X, bmf.FACTOR_W)]
    a.close()
    np.testing.assert_array_equal(mom[0][0], S1)
    assert (np.abs(mom[0][1] - S2) <= 4 * 2.0 ** -53 * np.abs(S2).max()).all()
    for sched in ((1, 1, 4, 0.0, 0, 0), (3, 2, 4, 0.0, 0, 0), (2, 1, 4, 0.0, 1, 0)):
        b, _ = _context(K, prec, sched)
        b.sweep(0, 3, None)
        Xb, Wb, _ = b.get_state(0)
        np.testing.assert_array_equal(Xb, X, err_msg=str(sched))
        np.testing.assert_array_equal(Wb, W, err_msg=str(sched))
        for f, want in zip((bmf.FACTOR_X, bmf.FACTOR_W), mom):
            got = b.get_moments(0, f)
            np.testing.assert_array_equal(got[0], want[0])
            np.testing.assert_array_equal(got[1], want[1])
        b.close()


def test_mixture_priors_are_factored_for_every_sweep():
    from paper_1703_00734_gb300 import bmf
    K = 9
    d = synth.make_workload(None, N=200, D=120, M=700, pattern="zipf", K=K, sigma=0.5, tau=4.0, seed=5, s_row=1.2,
                            s_col=1.2)
    out = []
    for split in (1, 4):
        m = bmf.BMF(d["N"], d["D"], d["row"], d["col"], d["val"], K, d["tau"], "fp32", I=2, J=2, X0=d["X0"],
                    W0=d["W0"], seed=3, summary="gmm", lam=12.0, components=3, max_samples=60)
        for stage in (1, 2):
            m.stage(stage, 60, None)
        for _ in range(split):
            m.stage(3, 12 // split, None)
        out.append(m.get_state(3)[:2])
        m.close()
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("K", [9, 16])
def test_priors_that_are_not_positive_definite(K):
    from paper_1703_00734_gb300 import bmf
    m, bad = _context(K, "fp32", (1, 1, 4, 0.0, 0, 0), bad=5)
    with pytest.raises(bmf.BmfError) as e:
        m.sweep(0, 2, None)
    assert e.value.status == 3 and f"arena row {bad})" in str(e.value)
    m.close()
