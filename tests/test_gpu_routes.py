"""Paths that the other bit-equality tests leave out, against one thread per chain: an
AxCaliberSMT tree of depth 4 with burn-in adaptation, slices well past the threshold that
selects them, and the 3-pool model's lane-split kernel where the library chooses it.
AxCaliberSMT, whose kernels read the constants of a model held in shared memory there, through the
server and the allocation-free entry point, whose results equal the sampler's bit for bit, and its
likelihoods in the ensemble sampler against the oracle."""
import numpy as np
import pytest
import torch

from conftest import make_voxels
from paper_2511_22094_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("samples", "mean", "std", "rhat", "accept_rate", "nonfinite", "step_scale")
ECHOES12 = tuple(2.0 + 4.0 * k for k in range(12))
CASES = {
    "axcal-tree-depth-4": (W.AXCAL_250K, 290, 4, dict(iterations=101, burnin=60, thin=10, adapt_window=6, adapt_target=0.25)),
    "axcal-many-slices": (W.AXCAL_250K, 25_001, 4, dict(iterations=1100, burnin=100, thin=50)),
    "axcal-slices-seven": (W.AXCAL_250K.with_(acq=W.AXCAL_250K.acq[:21]), 22_000, 4, dict(iterations=520, burnin=20, thin=50)),
    "mwi3-many-slices": (W.MWI3_1M, 23_000, 4, dict(iterations=1000, burnin=100, thin=50)),
    "mwi3-two-lanes": (W.MWI3_1M.with_(acq=ECHOES12), 4000, 2, dict(iterations=150, burnin=30, thin=20)),
}


@pytest.mark.parametrize("w,n,C,kw", CASES.values(), ids=CASES)
def test_same_bits_as_one_thread_per_chain(gac, orc, w, n, C, kw):
    mid = gac.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    th = W.truths(w, 0, n)
    sig = W.sigma(w, th)
    y = W.noisy_data(gac.forward_host(mid, th), W.noise(w, 0, n), sig)
    run = lambda **k: gac.run_host(mid, y, sig, n_chains=C, seed=4, **kw, **k)
    one, auto = run(lanes_per_chain=1), run()
    for k in KEYS:
        if one[k] is not None:
            np.testing.assert_array_equal(auto[k], one[k], err_msg=k)


@pytest.mark.parametrize("n_meas", [7, 16])
def test_axcal_on_every_entry_point(gac, orc, n_meas):
    w, n, C, I = W.AXCAL_250K.with_(acq=W.AXCAL_250K.acq[:3 * n_meas]), 700, 4, 300
    mid = gac.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    th, sig, y = make_voxels(orc, w, 0, n)
    want = gac.run_host(mid, y, sig, iterations=I, burnin=100, thin=20, n_chains=C, seed=9, lanes_per_chain=1)
    opts = gac.make_opts(I, 100, 20, C, 9)
    srv = gac.gac_server_create(4 << 30, 8)
    try:
        out = {k: np.zeros_like(want[k]) for k in ("mean", "std", "accept_rate")}
        gac.gac_server_wait(srv, gac.gac_server_submit(srv, mid, y, n, sig, 0.0, opts), 60.0, out)
    finally:
        gac.gac_server_destroy(srv)
    dev = {k: torch.zeros(want[k].shape, dtype=torch.float64 if k != "accept_rate" else torch.float32, device="cuda:0") for k in out}
    gac.gac_mcmc_run_noalloc(mid, torch.from_numpy(y).cuda(), n, torch.from_numpy(sig).cuda(), 0.0, None, opts, 70, dev,
                             torch.cuda.current_stream())
    for k in out:
        np.testing.assert_array_equal(out[k], want[k], err_msg=k)
        np.testing.assert_array_equal(dev[k].cpu().numpy(), want[k], err_msg=k)
    # the ensemble's likelihoods, of kept and of proposed states, against the oracle's model: the
    # tolerance of the library's own likelihood tests away from the posterior
    lb, ub = np.array(w.lb), np.array(w.ub)
    x0 = np.repeat(th[:, None, :], 20, axis=1) + 0.02 * (ub - lb) * np.random.default_rng(1).standard_normal((n, 20, len(lb)))
    x0 = np.clip(x0, lb + 1e-3 * (ub - lb), ub - 1e-3 * (ub - lb)).astype(np.float32)
    rec = gac.run_ensemble_host(mid, y, sig, iterations=40, burnin=0, thin=10, n_walkers=20, seed=2, x0=x0, trace_n_vox=6)["trace"]
    for v in range(6):
        for state, L in (("theta", "L"), ("prop", "Lp")):
            x, got = rec[v][state].reshape(-1, rec[v][state].shape[-1])[:, :4], rec[v][L].ravel()
            inside = np.isfinite(got) & (x >= lb).all(1) & (x <= ub).all(1)
            s64 = orc.forward(w.kind, w.acq, x[inside])
            want64 = -0.5 * (((y[v].astype(np.float64) - s64) / float(sig[v])) ** 2).sum(1)
            assert inside.mean() > 0.5
            assert (np.abs(got[inside] - want64) <= 1e-3 + 5e-5 * np.abs(want64)).all()
