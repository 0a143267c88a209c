"""Fits without a total-variation term take many updates in one launch.

Against the launch per update that coupled fits take: with a penalty far below
the rounding of every gradient (lambda 1e-25) that path computes the same FP32
values, so parameters are equal bit for bit and losses to the order of their
sums (1e-9).  Against the FP64 oracle: trajectory, losses and stopping iteration
of every model and loss, with a mask and weights; the rules stop inside, at the
end and in the first updates of a launch's chunk.
"""
import numpy as np
import pytest

from test_gpu_fit import LINEAR, MODELS, MONOEXP, MWI3, SMT, _problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("loss", [1, 2])
@pytest.mark.parametrize("kind,shape,iters", [(MWI3, (23, 11, 7), 140), (MONOEXP, (5, 5, 1), 257), (SMT, (40, 30, 11), 33),
                                               (LINEAR, (33, 1, 1), 16), (MWI3, (1, 1, 1), 3)])
@pytest.mark.parametrize("masked", [False, True])
def test_same_as_a_launch_per_update(gac, orc, kind, shape, iters, loss, masked):
    acq, lb, ub, y, theta0, mask, weight = _problem(orc, kind, shape=shape)
    mask[0] = 1
    mid = gac.gac_model_register(kind, acq, lb, ub, np.zeros(len(lb)))
    kw = dict(shape=shape, mask=mask if masked else None, weight=weight, loss=loss, iterations=iters, learning_rate=0.01)
    a_th, a_hist, a_done = gac.fit_host(mid, y, theta0, tv_lambda=1e-25, tv_params=1, **kw)
    b_th, b_hist, b_done = gac.fit_host(mid, y, theta0, **kw)
    assert a_done == b_done == iters
    np.testing.assert_array_equal(b_th, a_th)
    np.testing.assert_allclose(b_hist, a_hist, rtol=1e-9)
    if masked:
        np.testing.assert_array_equal(b_th[mask == 0], theta0[mask == 0])


@pytest.mark.parametrize("kind", [MONOEXP, MWI3, SMT, LINEAR])
@pytest.mark.parametrize("loss", [1, 2])
def test_fp64_follows_the_oracle(gac, orc, kind, loss):
    shape = (7, 6, 5)
    acq, lb, ub, y, theta0, mask, weight = _problem(orc, kind, shape=shape)
    mid = gac.gac_model_register(kind, acq, lb, ub, np.zeros(len(lb)))
    r_th, r_hist, r_done = orc.fit_run(kind, acq, lb, ub, y, theta0, shape=shape, mask=mask, weight=weight, loss=loss,
                                       iterations=60, lr=0.01, lam=0.0, tv_params=0, tv_dims=3)
    g_th, g_hist, g_done = gac.fit_host(mid, y, theta0, shape=shape, mask=mask, weight=weight, loss=loss, iterations=60,
                                        learning_rate=0.01, precision=gac.PREC_FP64)
    assert g_done == r_done == 60
    np.testing.assert_allclose(g_hist, r_hist, rtol=1e-9)
    assert (np.abs(g_th - r_th) <= 1e-6 * (ub - lb)).mean() >= 0.999


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("stop", [2, 20, 31, 32, 33, 64, 75])
def test_stops_where_the_losses_say(gac, orc, precision, stop):
    """The rules end the fit at the update the full history predicts, and the parameters are those
    of that update."""
    shape = (9, 8, 3)
    acq, lb, ub, y, theta0, mask, weight = _problem(orc, MONOEXP, shape=shape)
    mid = gac.gac_model_register(MONOEXP, acq, lb, ub, np.zeros(2))
    kw = dict(shape=shape, mask=mask, weight=weight, loss=2, learning_rate=0.002, precision=precision)
    _, hist, done = gac.fit_host(mid, y, theta0, iterations=100, **kw)
    assert done == 100 and (np.diff(hist[:80]) < 0).all()
    tol = 0.5 * (hist[stop - 1] + hist[stop - 2])
    want, want_hist, _ = gac.fit_host(mid, y, theta0, iterations=stop, **kw)
    th, h, d = gac.fit_host(mid, y, theta0, iterations=100, tol=tol, **kw)
    assert d == stop
    np.testing.assert_array_equal(th, want)
    np.testing.assert_array_equal(h, want_hist)
    window = 10
    slope = [abs(np.polyfit(np.arange(window), hist[t - window:t], 1)[0]) for t in range(window, 101)]
    cut = 0.5 * (slope[max(stop - window, 1)] + slope[max(stop - window, 1) - 1])
    want_stop = next(t for t, v in zip(range(window, 101), slope) if v < cut)
    _, _, d = gac.fit_host(mid, y, theta0, iterations=100, convergence_value=cut, convergence_window=window, **kw)
    assert d == want_stop
