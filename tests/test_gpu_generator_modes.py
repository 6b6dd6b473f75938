"""The device generator's numbers do not depend on the precision mode, and both forms of its normals
(tables up to K = 48, the FP64 functions above) are within their bounds of long double.

Tolerance of the functions' form, relative to the radius r of an element's pair: the angle 2 pi u2 is
rounded at 2^-51, the logarithm, the root, the sine or cosine and the product each within about one
unit of 2^-53, so 8 2^-53 r."""
import numpy as np
import pytest

from test_gpu_normals import _reference

pytestmark = pytest.mark.gpu


def _draws(K, N, seed, prec, t):
    from paper_1703_00734_gb300 import bmf
    m = bmf.BMF(N, 3, np.arange(3), np.arange(3), np.ones(3), K, 1.0, prec, seed=seed)
    z = m.generate_draws(t)
    m.close()
    return z


@pytest.mark.parametrize("K", [1, 8, 9, 16, 48, 49, 64])
def test_draws_do_not_depend_on_the_precision_mode(K):
    want = _draws(K, 701, 5, "fp64", 3)
    for prec in ("fp32", "bf16", "tf32"):
        np.testing.assert_array_equal(_draws(K, 701, 5, prec, 3), want, err_msg=prec)


@pytest.mark.parametrize("K,N,seed", [(49, 7, 1), (64, 20_000, 2 ** 63 + 5)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_normals_of_a_wide_model_are_within_their_bound(K, N, seed, prec):
    H = 2 * (K + K * (K - 1) // 2 + K)
    n = N * K // 2 * 2
    for t in (1, 7):
        z = _draws(K, N, seed, prec, t)[H:H + n]
        want = _reference(seed, t, 3, n)
        r = np.repeat(np.sqrt((want.reshape(-1, 2) ** 2).sum(1)), 2)
        assert (np.abs(z - want) <= 8 * 2.0 ** -53 * r).all()
