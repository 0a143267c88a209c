"""Problems of one to three waves of tiles, which run in slices (tiles take turns on the
GPU, the chains' state kept in device memory in between), against one launch
(which a traced run always takes): equal bit for bit.  Chain counts just past a
wave and in between, several chains a voxel, thinning grids that cross the
slices, burn-in adaptation, moments over every state and a start x0."""
import numpy as np
import pytest

from conftest import make_voxels
from paper_2511_22094_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("samples", "mean", "std", "rhat", "accept_rate", "nonfinite", "step_scale")
CASES = [(W.AXCAL_250K, 20_001, 4, dict(iterations=256, burnin=30, thin=16)),
         (W.AXCAL_250K, 13_000, 7, dict(iterations=301, burnin=100, thin=33, moments_mode=1, adapt_window=20, adapt_target=0.3)),
         (W.AXCAL_250K, 80_003, 1, dict(iterations=300, burnin=299, thin=100)),
         (W.MWI3_1M, 23_250, 4, dict(iterations=259, burnin=60, thin=17, adapt_window=7, adapt_target=0.25)),
         (W.MWI3_1M, 1300, 64, dict(iterations=256, burnin=0, thin=20))]


@pytest.mark.parametrize("w,n,C,kw", CASES, ids=[f"{c[0].name}-{c[1]}x{c[2]}" for c in CASES])
def test_slices_give_the_same_bits(gac, orc, w, n, C, kw):
    mid = gac.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    th = W.truths(w, 0, n)
    sig = W.sigma(w, th)
    y = W.noisy_data(gac.forward_host(mid, th), W.noise(w, 0, n), sig)
    y[3] = np.inf
    x0 = np.repeat(th[:, None, :], C, axis=1).astype(np.float32) if kw.get("moments_mode") else None
    run = lambda tr: gac.run_host(mid, y, sig, n_chains=C, seed=12, trace_n_vox=tr, x0=x0, **kw)
    one, sliced = run(1), run(0)
    for k in KEYS:
        if one[k] is not None:
            np.testing.assert_array_equal(sliced[k], one[k], err_msg=k)
    assert (one["nonfinite"][:, 3] == kw["iterations"]).all()
