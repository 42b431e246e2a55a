"""EXP3 fit (one cluster per observable that needs it) vs the oracle: the fewest
levels it takes, one and two levels per lane, one and several observables, and
the EXP_LOGLIN fallback that reaches it for some observables only."""
import numpy as np
import pytest

from oracle import fit as ofit
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", [ofit.M_EXP3, ofit.M_EXP_LOGLIN])
@pytest.mark.parametrize("nl,n_obs", [(1, 2), (2, 3), (3, 1), (5, 70), (32, 3), (33, 3), (64, 2)])
def test_exp3(nl, n_obs, method):
    require_gpu()
    from paper_2501_13237_gb300 import nne
    ctx = nne.Context(0)
    rng = np.random.default_rng(nl * 100 + n_obs)
    lams = np.linspace(1.0, 6.0, nl)
    y = (rng.uniform(0.3, 1, n_obs) * np.exp(-np.outer(lams, rng.uniform(0.1, 0.6, n_obs)))
         + rng.uniform(0.02, 0.05, n_obs))
    y *= 1 + 0.02 * rng.standard_normal(y.shape)
    if method == ofit.M_EXP_LOGLIN:
        y[1:, ::2] *= -1          # only the smallest level keeps its sign: the fallback
    lf = np.log(np.linspace(0.5, 0.999, nl))
    est, st = ctx.extrapolate(lams, y, lf, method=method, lambda_star=1.0)
    ref, rst = ofit.extrapolate(method, lams, y, 1.0, log_fid=lf)
    assert (st == rst).all()
    np.testing.assert_allclose(est, ref, rtol=0, atol=1e-7)
