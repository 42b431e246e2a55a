"""Expectation values of states whose site tensors lie far from order 1 (written with
nne_state_write_site; <P> = Tr(P rho)/Tr(rho) does not depend on their scale).  Two
neighbouring sites carry the same factor, so the stored per-site vectors of both are
that small or large and a two-site string multiplies them; at 1e36 the sums over a bond
leave float32's range as well.  Every one- and neighbouring two-site string and one of
three sites against the oracle's contraction."""
import numpy as np
import pytest

from oracle import mps
from tests.gpu_util import rand_c, require_gpu

pytestmark = pytest.mark.gpu
TOL = {1: 1e-11, 0: 2e-5}      # as the other sweep tests


def strings(n):
    codes = np.zeros((12 * n - 8, n), np.uint8)
    for i in range(n):
        for a in range(3):
            codes[3 * i + a, i] = a + 1
    for i in range(n - 1):
        for a in range(9):
            codes[3 * n + 9 * i + a, i:i + 2] = a // 3 + 1, a % 3 + 1
    codes[-1, 1:4] = 1, 2, 3
    return codes


@pytest.mark.parametrize("bonds", [[1, 4, 9, 12, 7, 4, 1], [1, 4, 16, 64, 66, 64, 16, 4, 1]])
@pytest.mark.parametrize("dtype,scale", [(0, 1e-38), (0, 1e-36), (0, 1e-25), (0, 1e-21), (0, 1e19), (0, 1e25),
                                         (0, 1e36), (1, 1e-100), (1, 1e100)])
@pytest.mark.parametrize("at", [0, 2])
def test_scaled_pair(bonds, dtype, scale, at):
    require_gpu()
    from paper_2501_13237_gb300 import nne
    n = len(bonds) - 1
    rng = np.random.default_rng(17)
    M = [rand_c(rng, (bonds[k], 4, bonds[k + 1])) for k in range(n)]
    for k in (at, at + 1):
        M[k] = M[k] * scale
    if dtype == 0:
        M = [m.astype(np.complex64) for m in M]
    st = nne.State(nne.Context(0), n, max(bonds), 1, dtype)
    for k in range(n):
        st.write_site(0, k, M[k])
    codes = strings(n)
    vals, _ = st.expect(codes)
    st.close()
    ref_st = mps.VMPO(n, max(bonds))
    ref_st.M = [m.astype(np.complex128) for m in M]
    # the oracle contracts in float64 without scaling: bring its tensors to order 1
    for k in (at, at + 1):
        ref_st.M[k] = ref_st.M[k] / scale
    ref = ref_st.expect_codes(codes)
    assert (np.abs(vals[0] - ref) <= TOL[dtype] * np.maximum(1.0, np.abs(ref))).all()


def test_environment_adds_no_rounding():
    """A chain of bonds 1 whose environments are real: every product has the factor 1, so the
    sweep's only error is the double-float scaling (2^-46 per site), not float32's rounding
    of a scaled environment."""
    require_gpu()
    from paper_2501_13237_gb300 import nne
    n = 24
    rng = np.random.default_rng(5)
    M = [rand_c(rng, (1, 4, 1)).astype(np.complex64) for _ in range(n)]
    for m in M:
        m[0, [0, 3], 0] = rng.uniform(0.1, 1.0, 2)
    st = nne.State(nne.Context(0), n, 4, 1, nne.C64)
    for k in range(n):
        st.write_site(0, k, M[k])
    codes = strings(n)
    vals, _ = st.expect(codes)
    st.close()
    ref_st = mps.VMPO(n, 4)
    ref_st.M = [m.astype(np.complex128) for m in M]
    ref = ref_st.expect_codes(codes)
    assert (np.abs(vals[0] - ref) <= 1e-12 * np.maximum(1.0, np.abs(ref))).all()
