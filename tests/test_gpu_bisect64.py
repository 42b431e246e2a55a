"""Eigenvalues of complex128 states' tridiagonal problems: the bracket ends at 2 eps_64 ||T||,
so the midpoint is within eps_64 ||T|| of the eigenvalue where the Sturm counts are exact --
diagonal matrices, whose minors' signs have no rounding.  One size per number of lanes that
share an eigenvalue (32, 16, 8, 4), several matrices, scales far from 1."""
import numpy as np
import pytest

from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu
EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("n,r", [(64, 64), (200, 65), (256, 192), (300, 300), (512, 321), (640, 640)])
@pytest.mark.parametrize("scale", [1.0, 1e-100, 1e100])
def test_bracket(n, r, scale):
    require_gpu()
    from tests import native
    lib = native.library("tri64")
    rng = np.random.default_rng(n + r)
    d = rng.uniform(-1, 1, (4, n))
    ref = -np.sort(-d, axis=1)[:, :r]
    lamf = np.ascontiguousarray(ref.astype(np.float32))
    # the float32 estimates are those of the matrix: they follow its scale only inside float32's range
    with np.errstate(over="ignore"):
        lamf = (lamf.astype(np.float64) * scale).astype(np.float32)
    d = np.ascontiguousarray(d * scale)
    e, lam = np.zeros((4, n)), np.zeros((4, r))
    p = lambda a: a.ctypes.data_as(native.ctypes.c_void_p)
    assert lib.bisect64_host(n, r, 4, p(d), p(e), p(lamf), p(lam)) == 0
    ref = -np.sort(-d, axis=1)[:, :r]
    norm = np.abs(d).max(axis=1, keepdims=True)
    assert (np.abs(lam - ref) <= 1.1 * EPS * norm).all()
