"""The device generator's normals against long double, element by element: streams that end inside
a call of four, the uniforms next to 0 and 1 that the generated words reach, every quadrant.

Tolerance: the logarithm, root, sine and cosine are each within one unit of 2^-53 of their leading
terms and the product adds a half, so |dz| <= 5 2^-53 max(1, |z|)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _reference(seed, t, tag, n):
    b = np.random.Philox(key=np.array([seed, 0], np.uint64))
    start = (t << 64) + (tag << 128) - 1          # numpy steps the counter before each call
    st = b.state
    st["state"]["counter"] = np.array([(start >> (64 * k)) & (2 ** 64 - 1) for k in range(4)], np.uint64)
    st["buffer_pos"] = 4
    b.state = st
    w = b.random_raw(-(-n // 4) * 4).reshape(-1, 4)
    LD = np.longdouble
    out = np.empty(w.shape, LD)
    for a in (0, 2):
        u1 = ((w[:, a] >> np.uint64(11)) + np.uint64(1)).astype(LD) / LD(2) ** 53
        u2 = (w[:, a + 1] >> np.uint64(11)).astype(LD) / LD(2) ** 53
        r, ang = np.sqrt(-2 * np.log(u1)), u2 * 2 * LD("3.14159265358979323846264338327950288419716939937510")
        out[:, a], out[:, a + 1] = r * np.cos(ang), r * np.sin(ang)
    return out.reshape(-1)[:n]


@pytest.mark.parametrize("K,N,seed", [(1, 5, 1), (3, 1001, 2), (16, 60_000, 2 ** 63 + 5)])
def test_normals_are_within_their_bound(K, N, seed):
    from paper_1703_00734_gb300 import bmf
    m = bmf.BMF(N, 3, np.arange(3), np.arange(3), np.ones(3), K, 1.0, "fp64", seed=seed)
    H = 2 * (K + K * (K - 1) // 2 + K)
    for t in (1, 7):
        z = m.generate_draws(t)[H:H + N * K]
        want = _reference(seed, t, 3, N * K)
        err = np.abs(z.astype(np.longdouble) - want) / np.maximum(1, np.abs(want))
        assert err.max() <= 5 * 2.0 ** -53, float(err.max())
    m.close()
