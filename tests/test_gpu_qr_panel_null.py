"""Gauge moves of site tensors of more than 160 rows whose columns are nearly or exactly null:
one large entry per column among rounding noise of many decades (pivots whose float32
squares are denormal), zero columns, equal columns, columns graded down to the square root
of float32's range.  The moved site is an isometry and the contraction of the three sites is
unchanged up to its norm, so the triangular factor is tested with it."""
import numpy as np
import pytest

from tests.gpu_util import rand_c, require_gpu

pytestmark = pytest.mark.gpu
TOL = {0: 2e-5, 1: 1e-12}      # as the other gauge moves


def tiny_noise(rng, shape, lo=1e-24, hi=1e-7):
    mag = np.exp(rng.uniform(np.log(lo), np.log(hi), shape))
    return mag * np.exp(2j * np.pi * rng.uniform(size=shape))


def matrix(kind, m, n, rng):
    if kind == "permuted":
        X = tiny_noise(rng, (m, n))
        X[rng.permutation(m)[:n], np.arange(n)] += rng.uniform(0.4, 0.6, n) * np.exp(2j * np.pi * rng.uniform(size=n))
        return X
    X = rand_c(rng, (m, n))
    if kind == "null":
        X[:, rng.permutation(n)[:n // 3]] = 0
    elif kind == "equal":
        X[:, 1::2] = X[:, 0::2][:, :X[:, 1::2].shape[1]]
    else:
        X *= 10.0 ** -np.linspace(0, 17, n)
    return X


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("direction", [+1, -1])
@pytest.mark.parametrize("dl,dr", [(41, 40), (60, 129), (128, 65), (200, 250)])
@pytest.mark.parametrize("kind", ["permuted", "null", "equal", "graded"])
def test_nearly_null_columns(kind, dl, dr, direction, dtype):
    require_gpu()
    from paper_2501_13237_gb300 import nne
    rng = np.random.default_rng(dl * 1000 + dr)
    X = matrix(kind, 4 * dl, dr, rng)
    M = X.reshape(dl, 4, dr) if direction > 0 else X.conj().T.reshape(dr, 4, dl)
    if direction < 0:
        dl, dr = dr, dl
    N, other = rand_c(rng, (dr, 4, 7)), rand_c(rng, (7, 4, 6))
    if direction < 0:
        N, other = rand_c(rng, (7, 4, dl)), rand_c(rng, (6, 4, 7))
    if dtype == 0:
        M, N, other = (a.astype(np.complex64) for a in (M, N, other))
    ctx = nne.Context(0)
    st = nne.State(ctx, 12, 256, 1, dtype)
    a = 5
    b = a + direction
    for k, T in ((a, M), (b, N), (b + direction, other)):
        st.write_site(0, k, T)
    st.set_centre(a)
    G = ctx.build_superops(np.stack([np.eye(4, dtype=complex)]), np.zeros((1, 4)))
    st.apply_layer([b if direction > 0 else b - 1], G, direction)
    out = [st.read_site(0, k).astype(complex) for k in (a, b, b + direction)]
    st.close()
    Q = out[0]
    k = Q.shape[2] if direction > 0 else Q.shape[0]
    iso = Q.reshape(-1, k) if direction > 0 else Q.reshape(k, -1).conj().T
    assert np.abs(iso.conj().T @ iso - np.eye(k)).max() < 10 * TOL[dtype]

    def whole(ts):
        ts = ts if direction > 0 else ts[::-1]
        T = np.einsum("asc,ctb->astb", ts[0], ts[1])
        T = np.einsum("astb,bud->astud", T, ts[2]).reshape(-1)
        return T / np.linalg.norm(T)

    assert np.linalg.norm(whole(out) - whole([t.astype(complex) for t in (M, N, other)])) < 10 * TOL[dtype]
