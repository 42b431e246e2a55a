"""QR panel shapes at their edges through the gauge moves (QR and LQ of a site
tensor): panel widths with remainders, rows per warp, CTAs per matrix, and the
border (160 rows) between the two panel kernels.  The state's contraction is
unchanged and the moved site is an isometry."""
import numpy as np
import pytest

from tests.gpu_util import rand_c, require_gpu

pytestmark = pytest.mark.gpu
TOL = {0: 2e-5, 1: 1e-12}      # complex64: some 100 eps of the tensor's norm; complex128 likewise


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("direction", [+1, -1])
@pytest.mark.parametrize("dl,dr", [(3, 5), (8, 32), (40, 40), (41, 40), (41, 33), (64, 31), (60, 129), (128, 65),
                                   (200, 250)])
def test_gauge_move(dl, dr, direction, dtype):
    require_gpu()
    from paper_2501_13237_gb300 import nne
    ctx = nne.Context(0)
    rng = np.random.default_rng(dl * 1000 + dr)
    if direction < 0:
        dl, dr = dr, dl
    st = nne.State(ctx, 12, 256, 1, dtype)
    M, N = rand_c(rng, (dl, 4, dr)), rand_c(rng, (dr, 4, 7) if direction > 0 else (7, 4, dl))
    a = 5                                          # moved site; its neighbour takes the factor
    b = a + direction
    st.write_site(0, a, M)
    st.write_site(0, b, N)
    st.set_centre(a)
    # a gate at the other side of the neighbour moves the centre there first
    other = rand_c(rng, (7, 4, 6) if direction > 0 else (6, 4, 7))
    st.write_site(0, b + direction, other)
    G = ctx.build_superops(np.stack([np.eye(4, dtype=complex)]), np.zeros((1, 4)))
    st.apply_layer([b if direction > 0 else b - 1], G, direction)
    Q = st.read_site(0, a).astype(np.complex128)
    k = Q.shape[2] if direction > 0 else Q.shape[0]
    iso = Q.reshape(-1, k) if direction > 0 else Q.reshape(k, -1).conj().T
    assert np.abs(iso.conj().T @ iso - np.eye(k)).max() < 10 * TOL[dtype]
    # the projection of M on the isometry is M itself
    X = M.reshape(-1, dr) if direction > 0 else M.reshape(dl, -1).conj().T
    assert np.linalg.norm(iso @ (iso.conj().T @ X) - X) < 10 * TOL[dtype] * np.linalg.norm(X)
    st.close()
