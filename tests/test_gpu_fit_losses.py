"""A fit's losses and parameters do not depend on the kernels that compute them: many updates a
launch, a list of the fitted voxels and the grid's kernel (which a penalty far below the rounding
of every gradient, or a tolerance that no loss meets, selects) give the same bits.  Grids of less
than a warp, of one and of several tiles a warp, ragged; more updates than one batch of losses."""
import numpy as np
import pytest

from test_gpu_fit import MONOEXP, MWI3, SMT, _problem

pytestmark = pytest.mark.gpu


def _big(orc, kind, shape, n_acq):
    """A small problem's voxels repeated over a grid, each with its own start."""
    n = int(np.prod(shape))
    acq, lb, ub, y, theta0, _, weight = _problem(orc, kind, shape=(31, 10, 5))
    if kind == MONOEXP and n_acq:
        acq, y = acq[:n_acq], y[:, :n_acq]
    rep = lambda a: np.ascontiguousarray(np.concatenate([a] * (n // len(a) + 1))[:n])
    u = np.random.default_rng(9).uniform(0.2, 0.8, (n, len(lb)))
    return acq, lb, ub, rep(y), lb + u * (ub - lb), rep(weight)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("kind,shape", [(MONOEXP, (9, 8, 3)), (MONOEXP, (37, 41, 9)), (SMT, (40, 30, 11)), (MWI3, (23, 11, 7)),
                                        (MONOEXP, (101, 97, 31)), (MWI3, (97, 101, 13))])
def test_many_updates_a_launch(gac, orc, kind, shape, precision):
    if precision == 2 and np.prod(shape) > 100_000 and kind == MWI3:
        shape = (60, 40, 9)
    acq, lb, ub, y, theta0, weight = _big(orc, kind, shape, 0)
    mid = gac.gac_model_register(kind, acq, lb, ub, np.zeros(len(lb)))
    mask = (np.random.default_rng(2).uniform(size=len(y)) < 0.7).astype(np.uint8)
    for m in (None, mask):
        kw = dict(shape=shape, mask=m, weight=weight, loss=2, iterations=20, learning_rate=0.01, precision=precision)
        a_th, a_hist, _ = gac.fit_host(mid, y, theta0, tv_lambda=1e-25, tv_params=1, tol=1e-300, **kw)
        for rules in (dict(), dict(tol=1e-300)):
            b_th, b_hist, _ = gac.fit_host(mid, y, theta0, **rules, **kw)
            np.testing.assert_array_equal(b_th, a_th)
            np.testing.assert_array_equal(b_hist, a_hist)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("kind,n_acq,tv_params", [(MONOEXP, 12, 0b11), (MONOEXP, 7, 0b10), (MWI3, 0, 0b1000001), (SMT, 0, 0b1)])
def test_list_of_fitted_voxels(gac, orc, kind, n_acq, tv_params, precision):
    """More than 97,280 fitted voxels: warps with a second tile, the last of them partial; rows of
    whole and of partial 16 bytes; one and two penalised maps; 130 updates."""
    shape, iterations = ((71, 53, 47), 130) if kind == MONOEXP else ((71, 53, 40), 30)
    acq, lb, ub, y, theta0, weight = _big(orc, kind, shape, n_acq)
    mask = (np.random.default_rng(5).uniform(size=len(y)) < 0.78).astype(np.uint8)
    assert 97_280 < mask.sum() <= 0.8 * len(mask) and mask.sum() % 32
    mid = gac.gac_model_register(kind, acq, lb, ub, np.zeros(len(lb)))
    kw = dict(shape=shape, mask=mask, weight=weight, loss=1, iterations=iterations, learning_rate=0.01, precision=precision,
              tv_lambda=0.02, tv_params=tv_params)
    a_th, a_hist, _ = gac.fit_host(mid, y, theta0, tol=1e-300, **kw)
    b_th, b_hist, _ = gac.fit_host(mid, y, theta0, **kw)
    np.testing.assert_array_equal(b_th, a_th)
    np.testing.assert_array_equal(b_hist, a_hist)
