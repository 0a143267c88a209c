"""Blocks of 128 threads (taken where they spread the chains more evenly over the
SMs) against blocks of 256 (which a traced run always takes): the results do not
depend on the tiling, so they are equal bit for bit."""
import numpy as np
import pytest

from conftest import make_voxels
from paper_2511_22094_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("samples", "mean", "std", "rhat", "accept_rate", "nonfinite", "step_scale")
CASES = [(W.MWI3_1M, 4801, 3), (W.MWI3_1M, 12_345, 4), (W.MWI3_1M, 50_000, 4), (W.SMT_1P5M, 12_345, 4),
         (W.AXCAL_250K, 7001, 7), (W.MONOEXP_4K, 700, 64), (W.MONOEXP_4K, 200_003, 1)]


@pytest.mark.parametrize("w,n,C", CASES, ids=[f"{c[0].name}-{c[1]}x{c[2]}" for c in CASES])
def test_half_blocks_give_the_same_bits(gac, orc, w, n, C):
    mid = gac.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    w = w.with_(n_vox=max(n, w.n_vox))
    th, sig, y = make_voxels(orc, w, 0, n)
    for prec in (gac.PREC_MIXED, gac.PREC_FP32):
        for kw in (dict(moments_mode=0), dict(moments_mode=1, adapt_window=6, adapt_target=0.3)):
            run = lambda tr: gac.run_host(mid, y, sig, iterations=24, burnin=12, thin=3, n_chains=C, seed=8, precision=prec,
                                          lanes_per_chain=1, trace_n_vox=tr, **kw)
            full, half = run(1), run(0)
            for k in KEYS:
                np.testing.assert_array_equal(half[k], full[k], err_msg=k)
