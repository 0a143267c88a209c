"""The speculative sampler kernel (several lanes a chain, each a node of the tree
of coming accept/reject decisions) against the one-thread kernel: it computes
the same values with the same functions, so every output is equal bit for bit.

Sizes reach each tree depth (5, 4, 3, 2 for about <= 600, <= 1,200, <= 2,400 or
4,800 and <= 19,000 chains), with iteration counts and adaptation windows that
end inside a round, partial blocks of echoes, several chains a voxel that leave
lanes over, thinning of 1, moments over every state, and a voxel without a finite
likelihood.
"""
import numpy as np
import pytest

from conftest import make_voxels
from paper_2511_22094_gb300 import workloads as W

pytestmark = pytest.mark.gpu

UNEVEN = (2.0, 3.0, 7.5, 11.0, 20.0, 33.0, 46.0)
KEYS = ("samples", "mean", "std", "rhat", "accept_rate", "nonfinite", "step_scale")

#: workload, acquisitions, voxels, chains, options
CASES = {
    "mwi3-d5-every-state-kept": (W.MWI3_1M, W.MWI3_1M.acq, 40, 3, dict(iterations=101, burnin=0, thin=1)),
    "mwi3-d4-partial-block": (W.MWI3_1M, W.MWI3_1M.acq[:22], 290, 4, dict(iterations=203, burnin=50, thin=7)),
    "mwi3-d3-adapt-all": (W.MWI3_1M, W.MWI3_1M.acq[:13], 500, 4,
                          dict(iterations=300, burnin=150, thin=9, adapt_window=20, adapt_target=0.3, moments_mode=1)),
    "mwi3-d2-uneven": (W.MWI3_1M, UNEVEN, 3000, 2, dict(iterations=77, burnin=11, thin=5)),
    "monoexp-d5-one-chain": (W.MONOEXP_4K, W.MONOEXP_4K.acq, 1, 1, dict(iterations=64, burnin=0, thin=2)),
    "monoexp-d4-all": (W.MONOEXP_4K, W.MONOEXP_4K.acq + (38.0,), 1100, 1,
                       dict(iterations=331, burnin=100, thin=3, moments_mode=1)),
    "monoexp-d3-adapt": (W.MONOEXP_4K, W.MONOEXP_4K.acq[:5], 701, 3,
                         dict(iterations=200, burnin=120, thin=4, adapt_window=7, adapt_target=0.4)),
    "monoexp-d2-uneven": (W.MONOEXP_4K, UNEVEN, 5000, 1, dict(iterations=90, burnin=9, thin=10)),
    "smt-d5-short": (W.SMT_1P5M, W.SMT_1P5M.acq, 33, 5, dict(iterations=3, burnin=0, thin=1)),
    "smt-d4": (W.SMT_1P5M, W.SMT_1P5M.acq, 300, 4, dict(iterations=150, burnin=30, thin=2)),
    "smt-d3-nine-b": (W.SMT_1P5M, (0.0, 1.0, 0.0, 2.5, 5.0, 7.5, 10.0, 3.0, 4.0), 1000, 4,
                      dict(iterations=100, burnin=20, thin=6, moments_mode=1)),
    "smt-d2-no-b0": (W.SMT_1P5M, (0.5, 1.0, 2.5, 5.0), 3000, 4, dict(iterations=60, burnin=10, thin=50)),
    "axcal-d5": (W.AXCAL_250K, W.AXCAL_250K.acq, 100, 4, dict(iterations=202, burnin=50, thin=10)),
    "axcal-d4-adapt": (W.AXCAL_250K, W.AXCAL_250K.acq[:21], 333, 3,
                       dict(iterations=100, burnin=60, thin=10, adapt_window=6, adapt_target=0.25)),
    "axcal-d3": (W.AXCAL_250K, W.AXCAL_250K.acq, 1100, 4, dict(iterations=50, burnin=10, thin=4)),
    "axcal-d2-64-chains": (W.AXCAL_250K, W.AXCAL_250K.acq, 5, 64, dict(iterations=60, burnin=10, thin=5, moments_mode=1)),
}


@pytest.mark.parametrize("case", CASES.values(), ids=CASES)
def test_same_bits_as_one_thread_per_chain(gac, orc, case):
    base, acq, n, C, kw = case
    w = base.with_(acq=tuple(acq))
    mid = gac.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    th, sig, y = make_voxels(orc, w, 0, n)
    if n > 20:
        y[17] = np.nan  # no finite likelihood: every proposal counted and rejected
    x0 = None
    if kw.get("moments_mode"):
        x0 = np.repeat(th[:, None, :], C, axis=1).astype(np.float32)
    run = lambda lanes: gac.run_host(mid, y, sig, n_chains=C, seed=31, voxel_base=5, x0=x0, lanes_per_chain=lanes, **kw)
    one, spec = run(1), run(0)
    for k in KEYS:
        if one[k] is not None:
            np.testing.assert_array_equal(spec[k], one[k], err_msg=k)
    if n > 20:
        assert (one["nonfinite"][:, 17] == kw["iterations"]).all()


def test_no_iterations_and_no_samples(gac, orc):
    """A round count of zero, and a burn-in that leaves no sample."""
    w = W.MWI3_1M
    mid = gac.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    th, sig, y = make_voxels(orc, w, 0, 7)
    for kw in (dict(iterations=0, burnin=0, thin=1), dict(iterations=40, burnin=40, thin=1),
               dict(iterations=40, burnin=10, thin=2**31 - 1)):
        one, spec = (gac.run_host(mid, y, sig, n_chains=2, seed=3, lanes_per_chain=k, **kw) for k in (1, 0))
        for k in KEYS:
            if one[k] is not None:
                np.testing.assert_array_equal(spec[k], one[k], err_msg=k)
        assert np.isnan(spec["mean"]).all()


@pytest.mark.parametrize("n,thin", [(2400, 3), (4800, 1), (4800, 4), (4096, 5)])
def test_monoexp_depth_follows_the_thinning(gac, orc, n, thin):
    """Two warps a scheduler at depth 4, and at depth 3 where thinning is short; the lane-split
    kernel otherwise: the same bits as one thread per chain."""
    w = W.MONOEXP_4K
    mid = gac.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    th, sig, y = make_voxels(orc, w.with_(n_vox=n), 0, n)
    run = lambda lanes: gac.run_host(mid, y, sig, iterations=120, burnin=17, thin=thin, n_chains=1, seed=6, lanes_per_chain=lanes)
    one, auto = run(1), run(0)
    for k in KEYS:
        np.testing.assert_array_equal(auto[k], one[k], err_msg=k)
