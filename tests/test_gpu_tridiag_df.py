"""Double-float reduction of the truncation's eigenproblem at the edges of its
launch shapes: 4 chi x 4 chi Gram matrices below the double-float sizes, of 256
and 512 threads, at the shared-memory limit (384) and above it (the first columns on rows in L2).
One complex64 gate step of a product gate with weak noise per size -- the middle
bond equals the kept rank, so the cut is gapped -- against the exact SVD update."""
import math

import numpy as np
import pytest

import workloads as wl
from oracle import mps
from tests.gpu_util import rand_c, require_gpu

pytestmark = pytest.mark.gpu
TOL = 1e-4     # complex64, as the other single-gate tests


def haar_u2(rng):
    q, r = np.linalg.qr(rand_c(rng, (2, 2)))
    return q * (np.diag(r) / np.abs(np.diag(r)))


@pytest.mark.parametrize("direction", [+1, -1])
@pytest.mark.parametrize("chi", [40, 41, 53, 64, 65, 96, 97, 110, 256])
def test_gate_step_sizes(chi, direction):
    require_gpu()
    from paper_2501_13237_gb300 import nne
    ctx = nne.Context(0)
    rng = np.random.default_rng(chi)
    A, B = rand_c(rng, (chi, 4, chi)), rand_c(rng, (chi, 4, chi))
    st = nne.State(ctx, 10, chi, 1, nne.C64)
    st.write_site(0, 4, A)
    st.write_site(0, 5, B)
    st.set_centre(4 if direction > 0 else 5)
    G = ctx.build_superops(np.stack([np.kron(haar_u2(rng), haar_u2(rng))]), np.array([[2e-3, 1e-3, 0.0, 0.0]]))
    st.apply_layer([4], G, direction)
    dims, _, ln, lf = st.info()
    left, right, f, nrm, s = mps.two_site_update(A, B, G.cpu().numpy()[0, 0], chi, direction)
    assert s[chi] < 0.2 * s[chi - 1]                   # gapped cut
    L, R = (st.read_site(0, k).astype(np.complex128) for k in (4, 5))
    got = np.einsum("asc,ctb->astb", L, R)
    ref = np.einsum("asc,ctb->astb", left, right)
    assert np.abs(got - ref).max() < TOL * max(1.0, np.abs(ref).max())
    assert abs(lf[0] - math.log(f)) < TOL and abs(ln[0] - math.log(nrm)) < TOL
    iso = L.reshape(-1, chi) if direction > 0 else R.reshape(chi, -1).conj().T
    assert np.abs(iso.conj().T @ iso - np.eye(chi)).max() < 10 * TOL
    st.close()
