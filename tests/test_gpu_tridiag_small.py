"""Float64 reduction of complex64 states' small eigenproblems (4 chi rows, up to 160) at
the edges of its launch shapes: fewer rows than CTAs, warps and lane groups with
remainders, the largest size.  Gate steps with a gapped cut against the exact SVD update."""
import math

import numpy as np
import pytest

from oracle import mps
from tests.gpu_util import rand_c, require_gpu

pytestmark = pytest.mark.gpu
TOL = 1e-4     # complex64, as the other single-gate tests


def haar_u2(rng):
    q, r = np.linalg.qr(rand_c(rng, (2, 2)))
    return q * (np.diag(r) / np.abs(np.diag(r)))


@pytest.mark.parametrize("chi", [1, 2, 4, 5, 8, 9, 24, 25, 33, 39, 40])
def test_gate_step_c64_small(chi):
    require_gpu()
    from paper_2501_13237_gb300 import nne
    ctx = nne.Context(0)
    rng = np.random.default_rng(chi)
    A, B = rand_c(rng, (chi, 4, chi)), rand_c(rng, (chi, 4, chi))
    st = nne.State(ctx, 10, chi, 1, nne.C64)
    st.write_site(0, 4, A)
    st.write_site(0, 5, B)
    st.set_centre(4)
    G = ctx.build_superops(np.stack([np.kron(haar_u2(rng), haar_u2(rng))]), np.array([[2e-3, 1e-3, 0.0, 0.0]]))
    st.apply_layer([4], G, +1)
    _, _, ln, lf = st.info()
    left, right, f, nrm, s = mps.two_site_update(A, B, G.cpu().numpy()[0, 0], chi, +1)
    assert s[chi] < 0.2 * s[chi - 1]
    L, R = (st.read_site(0, k).astype(np.complex128) for k in (4, 5))
    ref = np.einsum("asc,ctb->astb", left, right)
    assert np.abs(np.einsum("asc,ctb->astb", L, R) - ref).max() < TOL * max(1.0, np.abs(ref).max())
    assert abs(lf[0] - math.log(f)) < TOL and abs(ln[0] - math.log(nrm)) < TOL
    Lm = L.reshape(-1, chi)
    assert np.abs(Lm.conj().T @ Lm - np.eye(chi)).max() < 10 * TOL
    st.close()
