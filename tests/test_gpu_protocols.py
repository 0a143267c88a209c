"""Forward model and likelihood of SMT and AxCaliberSMT protocols at the edges of
the evaluation's blocks of six measurements, against the FP64 oracle: one to
thirteen b-values, b = 0 first, elsewhere, repeated or absent, and timings of one
to eight measurements.  Tolerances: the forward model's 1e-5 relative norm per
voxel; the likelihood's 5e-5 of its magnitude away from the posterior."""
import numpy as np
import pytest

from paper_2511_22094_gb300 import workloads as W

pytestmark = pytest.mark.gpu

B = (0.0, 1.0, 2.5, 5.0, 7.5, 10.0, 0.5, 3.0, 4.0, 6.0, 8.0, 9.0, 1.5)
SMT = {
    "b0-only": B[:1], "two": B[:2], "five": B[:5], "six": B[:6], "six-no-b0": B[1:7], "seven": B[:7],
    "twelve": B[:12], "thirteen": B, "b0-last": B[5::-1], "b0-twice": (0.0, 1.0, 0.0, 2.5, 5.0, 7.5),
    "seven-b0-second-block": B[1:7] + (0.0,),
}


def _axcal(n13, n30):
    b = [x for k in range(n13) for x in (0.3 + 0.6 * k, 13.0, 6.0)] + [x for k in range(n30) for x in (0.2 + 2.0 * k, 30.0, 6.0)]
    return tuple(b)


AXCAL = {f"{a}+{c}": _axcal(a, c) for a, c in ((1, 0), (2, 3), (6, 0), (6, 7), (8, 8), (5, 4))}
CASES = [(W.SMT_1P5M, k, v) for k, v in SMT.items()] + [(W.AXCAL_250K, k, v) for k, v in AXCAL.items()]


@pytest.mark.parametrize("w,name,acq", CASES, ids=[f"{c[0].name}-{c[1]}" for c in CASES])
def test_blocks_of_measurements(gac, orc, w, name, acq):
    n = 300
    mid = gac.gac_model_register(w.kind, acq, w.lb, w.ub, w.step)
    th = W.truths(w, 0, n).astype(np.float32).astype(np.float64)
    want = orc.forward(w.kind, acq, th)
    got = gac.forward_host(mid, th)
    rel = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
    assert rel.max() <= 1e-5
    sig = np.full(n, 0.02, np.float32)
    y = (want + 0.05 * np.random.default_rng(3).standard_normal(want.shape)).astype(np.float32)
    L = gac.loglik_host(mid, th, y, sig)
    L64 = -0.5 * (((y.astype(np.float64) - want) / sig[:, None].astype(np.float64)) ** 2).sum(1)
    assert (np.abs(L - L64) <= 1e-3 + 5e-5 * np.abs(L64)).all()


@pytest.mark.parametrize("kind", ["monoexp", "mwi3", "linear"])
@pytest.mark.parametrize("n_acq", [1, 2, 7, 33, 64])
def test_forward_rows(gac, orc, kind, n_acq):
    """Forward rows written by warps of 32 vectors: ragged counts, and rows shorter and longer
    than a warp, against the oracle (1e-5 relative norm) and against one vector at a time (equal)."""
    w = {"monoexp": W.MONOEXP_4K, "mwi3": W.MWI3_1M}.get(kind)
    acq = 2.0 + 0.7 * np.arange(n_acq)
    k, lb, ub = (W.LINEAR, (-2.0, -3.0), (2.0, 3.0)) if w is None else (w.kind, w.lb, w.ub)
    mid = gac.gac_model_register(k, acq, lb, ub, np.ones(len(lb)))
    rng = np.random.default_rng(n_acq)
    for n in (1, 31, 33, 1000):
        th = rng.uniform(lb, ub, (n, len(lb))).astype(np.float32).astype(np.float64)
        want, got = orc.forward(k, acq, th), gac.forward_host(mid, th)
        scale = np.linalg.norm(want, axis=1) if k != W.LINEAR else 4.0 + 3.0 * np.abs(acq).max()
        assert (np.linalg.norm(got - want, axis=1) <= 1e-5 * scale).all()
        for i in {0, n // 2, n - 1}:
            np.testing.assert_array_equal(gac.forward_host(mid, th[i])[0], got[i])


def test_forward_more_vectors_than_a_wave(gac, orc):
    w = W.MONOEXP_4K
    mid = gac.gac_model_register(w.kind, w.acq[:3], w.lb, w.ub, w.step)
    n = 200_001
    th = W.truths(w.with_(n_vox=n), 0, n).astype(np.float32).astype(np.float64)
    want, got = orc.forward(w.kind, w.acq[:3], th), gac.forward_host(mid, th)
    assert (np.linalg.norm(got - want, axis=1) <= 1e-5 * np.linalg.norm(want, axis=1)).all()
