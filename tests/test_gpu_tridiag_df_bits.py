"""The double-float reduction itself (complex64 states' eigenproblems of more than 160 rows),
through its launcher: an instance's result does not depend on what else is in the batch
(a single matrix takes clusters of 16 CTAs, eight take 12), and the reduction has float64
quality at the edges of its launch shapes: 256 and 512 threads, the shared-memory limit,
rows in L2, more than 1024 rows (a third kernel for the first columns), null columns,
matrices far from order 1."""
import numpy as np
import pytest

from tests.gpu_util import rand_c, require_gpu

pytestmark = pytest.mark.gpu


def reduce(H):
    from tests import native
    lib = native.library("tridiag_df")
    H = np.ascontiguousarray(H, np.complex64)
    b, n, _ = H.shape
    d, e, Vh = np.zeros((b, n)), np.zeros((b, n), complex), np.zeros((b, n, n), np.complex64)
    p = lambda a: a.ctypes.data_as(native.ctypes.c_void_p)
    assert lib.tridiag_df_host(n, b, p(H), p(d), p(e), p(Vh)) == 0
    return d, e, Vh


def grams(n, batch, kind, seed):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(batch):
        X = rand_c(rng, (n, n)) * np.exp(-4.0 * np.arange(n) / n)
        if kind == "null":          # rows and columns that are zero to the last bit
            X[n // 3:] = 0
        out.append(X @ X.conj().T / n * {"tiny": 1e-25, "huge": 1e25}.get(kind, 1.0))
    return np.array(out, np.complex64)


@pytest.mark.parametrize("n", [161, 256, 300, 380, 381, 640, 1030])
def test_result_does_not_depend_on_the_batch(n):
    require_gpu()
    H = grams(n, 8, "graded", n)
    d, e, Vh = reduce(H)
    for z in (0, 5):
        d1, e1, V1 = reduce(H[z:z + 1])
        assert (d1[0] == d[z]).all() and (e1[0, :-1] == e[z, :-1]).all() and (V1[0] == Vh[z]).all()


@pytest.mark.parametrize("n,kind", [(161, "graded"), (256, "graded"), (257, "graded"), (380, "graded"), (381, "graded"),
                                    (1024, "graded"), (1025, "graded"), (1028, "graded"), (1200, "graded"),
                                    (200, "null"), (380, "null"), (600, "null"), (1100, "null"),
                                    (200, "tiny"), (500, "tiny"), (200, "huge"), (500, "huge")])
def test_reduction_has_float64_quality(n, kind):
    require_gpu()
    H = grams(n, 2, kind, n)
    d, e, Vh = reduce(H)
    for z in range(2):
        A = np.tril(H[z].astype(complex))           # the lower triangle is read, the diagonal as real
        A = A + np.tril(A, -1).conj().T
        A[np.arange(n), np.arange(n)] = A.diagonal().real
        lam = np.linalg.eigvalsh(A)
        T = np.diag(d[z].astype(complex)) + np.diag(e[z, :-1], -1) + np.diag(e[z, :-1].conj(), 1)
        # backward error of a Householder reduction: at most about n units in the last place (2^-46)
        assert np.abs(np.linalg.eigvalsh(T) - lam).max() <= n * 2.0 ** -46 * np.abs(lam).max()
        # T = Q^H A Q, Q = P_0 P_1 ... from the float32 reflectors: n roundings of 2^-24
        B = A / np.abs(lam).max()
        for j in range(n - 2):
            v = Vh[z, j].astype(complex).conj()
            w = B @ v
            B -= 2 * np.outer(w, v.conj())
            B -= 2 * np.outer(v, v.conj() @ B)
        assert np.linalg.norm(B - T / np.abs(lam).max()) <= n * 2.0 ** -24 * np.linalg.norm(T) / np.abs(lam).max()
