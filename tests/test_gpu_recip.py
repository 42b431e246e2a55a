"""The kernels' own reciprocals and reciprocal square roots against exact arithmetic, at the
bounds their comments state, over the exponents their callers use: pivots and squared
norms from the null threshold (2^-1000 in float64) up, denormal squared norms in float32,
double-floats around order 1 and far from it."""
from fractions import Fraction

import numpy as np
import pytest

from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


def call(which, x):
    from tests import native
    lib = native.library("recip")
    x = np.ascontiguousarray(x, np.float64)
    y = np.zeros_like(x)
    p = lambda a: a.ctypes.data_as(native.ctypes.c_void_p)
    assert lib.recip_host(which, len(x), p(x), p(y)) == 0
    return y


def values(lo, hi, single, seed, count=20000):
    rng = np.random.default_rng(seed)
    m = rng.uniform(1.0, 2.0, count)
    if single:
        m = m.astype(np.float32).astype(float)
    x = np.ldexp(m, rng.integers(lo, hi, count))
    near = 1.0 + np.arange(-64, 65) * (2.0 ** -23 if single else 2.0 ** -52)
    x = np.r_[x, near, 2 * near, np.ldexp(1.0, np.arange(lo, hi + 1))]
    return x.astype(np.float32).astype(float) if single else x


def excess(x, y, power):
    """|1 - x y| for 1/x (power 1), |1 - x y^2| / 2 for 1/sqrt(x) (power 2): the relative error, to its square."""
    return max(float(abs(1 - Fraction(float(a)) * b ** power)) / power for a, b in zip(x, y))


@pytest.mark.parametrize("which,lo,hi,single,bound", [
    (0, -1000, 1000, False, 1.1 * 2.0 ** -53),
    (1, -999, 1000, False, 1.1 * 2.0 ** -53),
    (2, -148, 127, True, 2.0 ** -23),
])
def test_floats(which, lo, hi, single, bound):
    require_gpu()
    x = values(lo, hi, single, which)
    x = x[x > 0]
    y = [Fraction(float(v)) for v in call(which, x)]
    assert excess(x, y, 1 if which == 0 else 2) <= bound


@pytest.mark.parametrize("which,lo,hi,bound", [(3, -100, 100, 2.0 ** -44), (4, 0, 1, 2.0 ** -46)])
def test_double_floats(which, lo, hi, bound):
    require_gpu()
    hi_part = values(lo, hi, True, which)
    if which == 4:
        hi_part = hi_part[(hi_part >= 1) & (hi_part < 2)]
    rng = np.random.default_rng(9)
    lo_part = (hi_part * 2.0 ** -25 * rng.uniform(-1, 1, len(hi_part))).astype(np.float32).astype(float)
    x = np.stack([hi_part, lo_part], 1)
    y = call(which, x)
    xs = [Fraction(float(a)) + Fraction(float(b)) for a, b in x]
    ys = [Fraction(float(a)) + Fraction(float(b)) for a, b in y]
    power = 2 if which == 3 else 1
    assert max(float(abs(1 - a * b ** power)) / power for a, b in zip(xs, ys)) <= bound
