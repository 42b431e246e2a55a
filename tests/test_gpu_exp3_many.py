"""EXP3 fits of large tables: clusters take several observables at a time, and a thread
forms an observable's golden section instead of a warp where a cluster has more than eight
of them.  The estimates are those of small calls (one observable per cluster) to the bit,
whatever observables around them need EXP3, and those of the oracle."""
import numpy as np
import pytest

from oracle import fit as ofit
from tests.gpu_util import require_gpu

pytestmark = pytest.mark.gpu


def table(nl, n_obs, seed):
    rng = np.random.default_rng(seed)
    lams = np.linspace(1.0, 6.0, nl)
    y = (rng.uniform(0.3, 1, n_obs) * np.exp(-np.outer(lams, rng.uniform(0.1, 0.6, n_obs)))
         + rng.uniform(0.02, 0.05, n_obs))
    return lams, y * (1 + 0.02 * rng.standard_normal(y.shape)), np.log(np.linspace(0.5, 0.999, nl))


# 608 clusters: 608 and 609 are one and two observables per cluster, 5472 and 5473 nine and
# ten, 77824 and 77825 the full 128 and the first second pass
@pytest.mark.parametrize("n_obs", [608, 609, 4864, 5473, 12160, 77825])
@pytest.mark.parametrize("share", [1.0, 0.3])
def test_large_tables(n_obs, share):
    require_gpu()
    from paper_2501_13237_gb300 import nne
    ctx = nne.Context(0)
    lams, y, lf = table(4, n_obs, n_obs)
    method = ofit.M_EXP3
    if share < 1:
        method = ofit.M_EXP_LOGLIN
        flip = np.random.default_rng(1).random(n_obs) < share
        flip[:64] = True                    # a run of neighbours
        y[1:, flip] *= -1                   # the fallback
    est, st = ctx.extrapolate(lams, y, lf, method=method, lambda_star=1.0)
    pick = np.unique(np.r_[np.arange(0, 40), np.linspace(0, n_obs - 1, 500).astype(int), n_obs - 1])
    small, sst = ctx.extrapolate(lams, y[:, pick], lf, method=method, lambda_star=1.0)
    assert (st[pick] == sst).all() and (st == 0).all()
    assert (est[pick] == small).all()
    few = pick[::25]
    ref, _ = ofit.extrapolate(method, lams, y[:, few], 1.0, log_fid=lf)
    np.testing.assert_allclose(est[few], ref, rtol=0, atol=1e-7)


def test_too_few_levels_in_a_large_table():
    """Two levels: no EXP3 fit, the value at lambda* -- for every observable of a cluster."""
    require_gpu()
    from paper_2501_13237_gb300 import nne
    lams, y, lf = table(2, 9000, 3)
    est, st = nne.Context(0).extrapolate(lams, y, lf, method=ofit.M_EXP3, lambda_star=1.0)
    assert (st == -6).all() and (est == y[0]).all()


@pytest.mark.parametrize("n_obs", [1363, 1364, 5000])
@pytest.mark.parametrize("given", [False, True])
def test_tables_around_the_staged_size(n_obs, given):
    """4 levels of 1363 observables (with their y_zero) are the last to go over in one 64 KB
    copy: the same estimates above and below, with and without the optional inputs."""
    require_gpu()
    from paper_2501_13237_gb300 import nne
    ctx = nne.Context(0)
    lams, y, lf = table(4, n_obs, 7)
    opt = dict(log_fid=lf, y_zero=y[0]) if given else {}
    for method, tol in [(ofit.M_POLY, 1e-10), (ofit.M_EXP_LOGLIN, 1e-10)]:
        est, st = ctx.extrapolate(lams, y, method=method, degree=2, lambda_star=1.0, **opt)
        few = np.r_[0:20, n_obs - 20:n_obs]
        sub = dict(log_fid=lf, y_zero=y[0, few]) if given else {}
        ref, rst = ofit.extrapolate(method, lams, y[:, few], 1.0, degree=2, **sub)
        assert (st[few] == rst).all() and (st == 0).all()
        assert (np.abs(est[few] - ref) <= tol).all()
