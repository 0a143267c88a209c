"""The library's host side on a stand-in for the CUDA runtime (fake_gpu.py): what a call
launches, and what it does where a call of the runtime fails."""
import ctypes as ct

import numpy as np
import pytest

import fake_gpu
from paper_2511_22094_gb300 import workloads as W


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_gpu.load(tmp_path_factory.mktemp("fake"))


def _sampler(fake, w, n, C, **kw):
    """A run of zeros; returns the recorded launches."""
    g, gpu = fake
    mid = g.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    y = np.zeros((n, g.gac_model_info(mid)[1]), np.float32)
    g.run_host(mid, y, None, sigma_scalar=1.0, n_chains=C, seed=1, want_samples=False, **kw)
    return gpu.launches


@pytest.mark.parametrize("iterations", [256, 1000, 999_983, 2**31 - 48, 2**31 - 24, 2**31 - 2])
@pytest.mark.parametrize("w,n", [(W.AXCAL_250K, 20_001), (W.AXCAL_250K, 25_001), (W.MWI3_1M, 23_250)])
def test_slices_cover_every_iteration_of_every_tile(fake, w, n, iterations):
    """The launches of a run in slices take positions 0 .. count n_tiles - 1 in order, and the last
    slice ends at the last iteration, up to the largest iteration count that a call may have."""
    _, gpu = fake
    gpu.reset()
    seen = []

    def on_launch(name, args):
        at = lambda i, t: ct.cast(args[i], ct.POINTER(t)).contents.value
        seen.append((at(3, ct.c_int64), at(4, ct.c_int)))

    gpu.on_launch = on_launch
    launches = _sampler(fake, w, n, 4, iterations=iterations, burnin=0, thin=max(16, iterations - 1))
    assert {x[0] for x in launches} == {f"mh_slice_kernel<{w.kind}>"}
    n_tiles, q = (n + 63) // 64, seen[0][1]
    count = -(-iterations // q)
    assert 64 <= q and 2 <= count <= 24
    end = 0
    for (pos, qi), (_, grid, _, block, _) in zip(seen, launches):
        assert (pos, qi, block) == (end, q, 256) and 1 <= grid <= n_tiles
        end += grid
    assert end == count * n_tiles
