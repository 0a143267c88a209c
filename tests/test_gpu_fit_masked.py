"""Coupled fits (total variation) over a mask, as flags on a small grid and as a list of
its voxels on a grid of more tiles than the GPU holds warps.

Masks that leave tiles of 32 empty, ragged or full and single voxels: the small
grid against the FP64 oracle; the same voxels inside a large grid, whose other
voxels hold NaN, against the small grid: the fitted voxels and their neighbours are
the same, so parameters are equal bit for bit and losses to the order of their
sums.
"""
import numpy as np
import pytest

from test_gpu_fit import MODELS, MONOEXP, MWI3, _problem

pytestmark = pytest.mark.gpu


def _masks(shape, rng):
    n = int(np.prod(shape))
    z, y, x = np.meshgrid(*[np.linspace(-1, 1, k) for k in shape[::-1]], indexing="ij")
    ball = (x**2 + y**2 + z**2 < 0.9).ravel()
    one = np.zeros(n, bool)
    one[n // 2] = True
    last = np.zeros(n, bool)
    last[-1] = last[0] = True
    return {"ball": ball, "one": one, "ends": last, "sparse": rng.uniform(size=n) < 0.05, "dense": rng.uniform(size=n) < 0.97}


@pytest.mark.parametrize("name", ["ball", "one", "ends", "sparse", "dense"])
@pytest.mark.parametrize("kind", [MONOEXP, MWI3])
def test_masked_coupled_fit(gac, orc, kind, name):
    shape = (21, 17, 9)
    acq, lb, ub, y, theta0, _, weight = _problem(orc, kind, shape=shape)
    mask = _masks(shape, np.random.default_rng(4))[name].astype(np.uint8)
    mid = gac.gac_model_register(kind, acq, lb, ub, np.zeros(len(lb)))
    kw = dict(loss=1, tv_lambda=0.02, tv_params=0b11, learning_rate=0.01)
    r_th, r_hist, _ = orc.fit_run(kind, acq, lb, ub, y, theta0, shape=shape, mask=mask, weight=weight, loss=1, iterations=12,
                                  lr=0.01, lam=0.02, tv_params=0b11, tv_dims=3)
    g_th, g_hist, _ = gac.fit_host(mid, y, theta0, shape=shape, mask=mask, weight=weight, iterations=12,
                                   precision=gac.PREC_FP64, **kw)
    np.testing.assert_allclose(g_hist, r_hist, rtol=1e-9)
    assert (np.abs(g_th - r_th) <= 1e-6 * (ub - lb)).mean() >= 0.999
    np.testing.assert_array_equal(g_th[mask == 0], theta0[mask == 0])
    # the same voxels inside a large grid
    big = (64, 50, 40)

    def put(a, fill):
        out = np.full((big[2], big[1], big[0]) + a.shape[1:], fill, a.dtype)
        out[11:11 + shape[2], 2:2 + shape[1], 13:13 + shape[0]] = a.reshape((shape[2], shape[1], shape[0]) + a.shape[1:])
        return out.reshape((-1,) + a.shape[1:])

    inside = put(mask, 0) != 0
    for precision in (gac.PREC_FP32, gac.PREC_FP64):
        a_th, a_hist, _ = gac.fit_host(mid, y, theta0, shape=shape, mask=mask, weight=weight, iterations=40, precision=precision, **kw)
        b_th, b_hist, _ = gac.fit_host(mid, put(y, np.nan), put(theta0, 1e30), shape=big, mask=put(mask, 0),
                                       weight=put(weight, np.nan), iterations=40, precision=precision, **kw)
        np.testing.assert_array_equal(b_th[inside], a_th[mask != 0])
        assert (b_th[~inside] == put(theta0, 1e30)[~inside]).all()
        np.testing.assert_allclose(b_hist, a_hist, rtol=1e-9)
