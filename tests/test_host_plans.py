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


def _echoes(n):
    return W.MWI3_1M.with_(acq=tuple(2.0 + 0.7 * k for k in range(n)))


def _forward(fake, n_acq, n):
    g, _ = fake
    w = _echoes(n_acq)
    g.forward_host(g.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step), np.tile(w.ub, (n, 1)))


def _fit(fake, w, shape, **kw):
    g, _ = fake
    mid = g.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    n = int(np.prod(shape))
    return g.fit_host(mid, np.zeros((n, g.gac_model_info(mid)[1]), np.float32), np.tile(w.ub, (n, 1)), shape=shape, **kw)


def _ensemble(fake, w, n):
    g, _ = fake
    mid = g.gac_model_register(w.kind, w.acq, w.lb, w.ub, w.step)
    g.run_ensemble_host(mid, np.zeros((n, g.gac_model_info(mid)[1]), np.float32), None, sigma_scalar=1.0, iterations=10,
                        burnin=0, thin=5, n_walkers=20, seed=1)


def _run(w, n, C, **kw):
    return lambda fake: _sampler(fake, w, n, C, iterations=300, burnin=0, thin=100, **kw)


#: calls that launch the same kernel with more, then with less shared memory
SAME_KERNEL = {
    "forward": (lambda f: _forward(f, 64, 100), lambda f: _forward(f, 48, 100)),
    "sampler": (_run(_echoes(64), 100_000, 4), _run(_echoes(6), 100_000, 4)),
    "sampler-slices": (_run(_echoes(64), 23_250, 4), _run(_echoes(24), 23_250, 4)),
    "sampler-lanes": (_run(_echoes(24), 3000, 1, lanes_per_chain=4), _run(_echoes(18), 300, 1, lanes_per_chain=4)),
    "sampler-tree": (_run(_echoes(64), 301, 4), _run(_echoes(6), 290, 4)),
    "ensemble": (lambda f: _ensemble(f, _echoes(64), 100), lambda f: _ensemble(f, _echoes(6), 100)),
    "fit": (lambda f: _fit(f, _echoes(24), (9, 8, 7), iterations=20), lambda f: _fit(f, _echoes(12), (9, 8, 7), iterations=20)),
    "fit-tv": (lambda f: _fit(f, _echoes(24), (9, 8, 7), iterations=20, tv_lambda=0.1, tv_params=1),
               lambda f: _fit(f, _echoes(12), (9, 8, 7), iterations=20, tv_lambda=0.1, tv_params=1)),
}


@pytest.mark.parametrize("calls", SAME_KERNEL.values(), ids=SAME_KERNEL)
def test_another_threads_smaller_launch_does_not_fail_a_larger_one(fake, calls):
    """The kernels' shared-memory limits are the process's: a call with less between another
    call's settings and its launches leaves those as they are."""
    _, gpu = fake
    large, small = calls
    gpu.reset()
    small(fake)
    names = set(gpu.names())
    gpu.reset()
    inside = []

    def on_limit(name):
        if name not in inside:
            inside.append(name)
            small(fake)

    gpu.on_limit = on_limit
    large(fake)  # a launch past the kernel's limit fails
    assert inside and names <= set(gpu.names())
    for name in names:
        assert len({v for k, v in gpu.limits if k == name}) <= 1


def _count(gpu, kernel):
    return sum(n.startswith(kernel) for n in gpu.names())


@pytest.mark.parametrize("kernel,launch", [("fit_many", 1), ("fit_losses", 1), ("fit_many", 2), ("fit_losses", 2)])
@pytest.mark.parametrize("tol", [0.0, 1e-300])
def test_a_fit_whose_launch_fails_reports_it(fake, kernel, launch, tol):
    """Also where the failure is a want of memory: the updates before it have changed the state in
    place, so no other path may start from it."""
    g, gpu = fake
    gpu.reset()
    gpu.on_launch = lambda name, args: fake_gpu.OOM if name.startswith(kernel) and _count(gpu, kernel) == launch else 0
    with pytest.raises(g.GacError) as err:
        _fit(fake, _echoes(12), (9, 8, 7), iterations=300, tol=tol)
    assert err.value.status == 4 and _count(gpu, "fit_step") == 0 and gpu.in_use == 0


def test_a_fit_without_memory_for_its_saved_state(fake):
    """Stopping rules keep the state of before a launch of many updates; without memory for it
    every update is a launch, from the first on."""
    _, gpu = fake
    shape, n = (9, 8, 7), 504
    gpu.reset()
    _fit(fake, _echoes(12), shape, iterations=70, tol=1e-300)
    assert _count(gpu, "fit_many") == 3
    assert 3 * n * 9 * 4 in gpu.sizes
    peak = gpu.peak
    gpu.reset()
    gpu.memory = peak - 1
    _fit(fake, _echoes(12), shape, iterations=70, tol=1e-300)
    assert _count(gpu, "fit_many") == 0 and _count(gpu, "fit_step") == 70 and gpu.in_use == 0


@pytest.mark.parametrize("name", ["uncoupled", "uncoupled-masked", "uncoupled-rules", "tv-masked"])
def test_a_fit_runs_in_the_memory_that_a_launch_per_update_needs(fake, name):
    """The list of voxels, the loss shares and the saved state are extras: a call that has no room for
    them beside the work arrays does without, wherever the room ends."""
    _, gpu = fake
    tv = dict(tv_lambda=0.1, tv_params=1)
    shape = (64, 50, 40) if name == "tv-masked" else (40, 30, 11)
    n = int(np.prod(shape))
    kw = dict(iterations=50, tol=1e-300 if name == "uncoupled-rules" else 0.0)
    if "masked" in name:
        kw["mask"] = (np.arange(n) % 3 != 0).astype(np.uint8)
    plain = {**kw, **tv, "tol": 1e-300}
    if name == "tv-masked":
        kw.update(tv)
    run = lambda **k: (gpu.reset(), setattr(gpu, "memory", k.pop("memory", None)), _fit(fake, W.MONOEXP_4K, shape, **k))
    run(**plain)
    least = gpu.peak
    assert _count(gpu, "fit_step") == 50
    run(**kw)
    most = gpu.peak
    assert most > least and _count(gpu, "fit_step") == 0
    for memory in np.linspace(least, most, 33).astype(int):
        run(**kw, memory=memory)
        assert _count(gpu, "theta_to_u") == 1 and gpu.in_use == 0
        assert (_count(gpu, "fit_step") == 50) == (memory < most)
    with pytest.raises(fake[0].GacError) as err:
        run(**kw, memory=least - 100_000)
    assert err.value.status == 4 and gpu.in_use == 0


@pytest.mark.parametrize("n,updates", [(504, 128), (345_000, 48), (4_000_003, 4), (8_388_608, 2)])
def test_losses_of_few_updates_are_summed_by_the_whole_gpu(fake, n, updates):
    """The 64 MB of loss shares hold few updates of a large grid; the launch that sums them fills
    the SMs all the same."""
    _, gpu = fake
    gpu.reset()
    w = W.MONOEXP_4K.with_(acq=(2.0, 5.0))
    _fit(fake, w, (n, 1, 1), iterations=2 * updates)
    losses = [x for x in gpu.launches if x[0].startswith("fit_losses")]
    assert [x[2] for x in losses] == [updates] * 2
    for _, grid, count, block, _ in losses:
        assert grid * count * block // 32 >= min(8 * 152, n)


@pytest.mark.parametrize("w,precision,n,kernel", [
    (W.MONOEXP_4K, 1, 97_280, "fit_many"), (W.MONOEXP_4K, 1, 97_281, "fit_step"), (W.MONOEXP_4K, 2, 100, "fit_step"),
    (W.MWI3_1M, 1, 72_960, "fit_many"), (W.MWI3_1M, 1, 72_961, "fit_step")])
def test_stopping_rules_run_few_updates_past_the_stop(fake, w, precision, n, kernel):
    """A launch of many updates runs past a stop: only where that costs less than the idle launches
    it saves, in FP32 with at most one tile a warp (3-pool: a tile for three warps of four)."""
    _, gpu = fake
    for rules in (dict(tol=1e-300), dict(convergence_value=1e-300)):
        for extra in (0, 1000):  # voxels outside the mask
            mask = np.r_[np.ones(n, np.uint8), np.zeros(extra, np.uint8)]
            gpu.reset()
            _fit(fake, w, (n + extra, 1, 1), mask=mask, iterations=33, precision=precision, **rules)
            fits = [x.split("_kernel")[0] for x in gpu.names() if x.startswith(("fit_many", "fit_step", "fit_list"))]
            assert fits == [kernel] * (2 if kernel == "fit_many" else 33)


@pytest.mark.parametrize("n,inside,kernel", [(8_388_608, 1.0, "fit_many"), (8_388_609, 1.0, "fit_step"), (8_388_609, 0.5, "fit_many")])
def test_large_grids_take_the_grids_kernel(fake, n, inside, kernel):
    """Single updates a launch (the shares of two pass 64 MB) only where they skip voxels."""
    _, gpu = fake
    gpu.reset()
    mask = None if inside == 1.0 else (np.arange(n) % 2).astype(np.uint8)
    _fit(fake, W.MONOEXP_4K.with_(acq=(2.0, 5.0)), (n, 1, 1), iterations=20, mask=mask)
    fits = [x.split("_kernel")[0] for x in gpu.names() if x.startswith(("fit_many", "fit_step", "fit_list"))]
    assert fits == [kernel] * (10 if n == 8_388_608 else 20)


@pytest.mark.parametrize("tv,n,many_from", [(0.0, 1000, 1), (0.0, 128_000, 2), (0.1, 128_000, 3)])
def test_fits_of_few_updates(fake, tv, n, many_from):
    """One update of many voxels and one or two with a list take the grid's kernel, and the loss
    shares are sized for the updates there are."""
    _, gpu = fake
    mask = (np.arange(n) % 5 > 0).astype(np.uint8)
    for iterations in (1, 2, 3):
        gpu.reset()
        _fit(fake, W.MONOEXP_4K, (n, 1, 1), iterations=iterations, mask=mask, tv_lambda=tv, tv_params=1 if tv else 0)
        assert _count(gpu, "fit_step") == (iterations if iterations < many_from else 0)
        assert (4 * n * iterations in gpu.sizes) == (iterations >= many_from)



def _spec_cases():
    from test_gpu_spec import CASES
    return [pytest.param(name, *c, id=name) for name, c in CASES.items()]


@pytest.mark.parametrize("name,base,acq,n,C,kw", _spec_cases())
def test_speculative_cases_run_the_tree_they_name(fake, name, base, acq, n, C, kw):
    _, gpu = fake
    gpu.reset()
    _sampler(fake, base.with_(acq=tuple(acq)), n, C, **kw)
    depth = int(name.split("-d")[1][0])
    if name == "axcal-d4-adapt":  # 999 chains, three a voxel: 666 warps at depth 4 (a case of 4: test_gpu_routes.py)
        depth = 3
    assert gpu.names() == [f"mh_spec_kernel<{base.kind},{depth},{kw.get('moments_mode', 0)}>"]


def test_slice_and_tile_cases_run_slices_and_half_blocks(fake):
    """The sizes that the bit-equality tests of those kernels choose do reach them."""
    import test_gpu_slices
    import test_gpu_tiles
    _, gpu = fake
    for w, n, C, kw in test_gpu_slices.CASES:
        gpu.reset()
        _sampler(fake, w, n, C, **kw)
        assert set(gpu.names()) == {f"mh_slice_kernel<{w.kind}>"} and len(gpu.names()) > 2
    half = []
    for w, n, C in test_gpu_tiles.CASES:
        gpu.reset()
        _sampler(fake, w, n, C, iterations=24, burnin=12, thin=3, lanes_per_chain=1)
        half.append(gpu.names() == [f"mh_kernel<{w.kind},0,0,128>"])
    assert sum(half) >= len(half) - 1


#: workload, echoes or b-values, chains, thinning, moments over every state -> kernel
ROUTES = [
    # 3-pool, two blocks of echoes: two lanes a chain where moments are rare
    ("mwi3", 12, 4864, 100, 0, "mh_spec_kernel<2,2,0>"), ("mwi3", 12, 5000, 100, 0, "mh_split_kernel<2,2,0>"),
    ("mwi3", 12, 9728, 12, 0, "mh_split_kernel<2,2,0>"), ("mwi3", 12, 9728, 11, 0, "mh_spec_kernel<2,2,0>"),
    ("mwi3", 7, 14_000, 3, 0, "mh_split_kernel<2,2,0>"), ("mwi3", 12, 14_000, 2, 0, "mh_kernel<2,0,0,128>"),
    ("mwi3", 12, 19_000, 8, 0, "mh_split_kernel<2,2,0>"), ("mwi3", 12, 19_000, 7, 0, "mh_kernel<2,0,0,128>"),
    ("mwi3", 12, 9728, 100, 1, "mh_spec_kernel<2,2,1>"), ("mwi3", 13, 9728, 100, 0, "mh_spec_kernel<2,2,0>"),
    ("mwi3", 24, 14_000, 100, 0, "mh_kernel<2,0,0,128>"),
    # mono-exponential where the lane-split kernel does not apply: four warps a scheduler or three
    ("monoexp", 6, 19_000, 100, 0, "mh_spec_kernel<1,2,0>"), ("monoexp", 5, 19_000, 100, 0, "mh_kernel<1,0,0,128>"),
    ("monoexp", 5, 14_000, 100, 0, "mh_spec_kernel<1,2,0>"), ("monoexp", 5, 19_000, 4, 0, "mh_spec_kernel<1,2,0>"),
    ("monoexp", 30, 19_000, 100, 1, "mh_kernel<1,0,0,128>"), ("monoexp", 48, 19_000, 100, 0, "mh_spec_kernel<1,2,0>"),
    # the lane-split kernel, and trees with short thinning
    ("monoexp", 12, 2400, 3, 0, "mh_spec_kernel<1,4,0>"), ("monoexp", 12, 4800, 4, 0, "mh_spec_kernel<1,3,0>"),
    ("monoexp", 12, 4096, 5, 0, "mh_split_kernel<1,2,0>"), ("monoexp", 24, 9600, 5, 0, "mh_split_kernel<1,4,0>"),
    # blocks of 128 past one block an SM where the waves promise enough
    ("monoexp", 12, 200_000, 100, 0, "mh_kernel<1,0,0,128>"), ("monoexp", 12, 240_000, 100, 0, "mh_kernel<1,0,0,256>"),
    ("monoexp", 12, 400_000, 100, 0, "mh_kernel<1,0,0,256>"), ("smt", 6, 393_216, 100, 0, "mh_kernel<3,0,0,128>"),
    ("mwi3", 24, 200_000, 100, 0, "mh_kernel<2,0,0,128>"),
    # SMT protocols of fewer than six b-values
    ("smt", 5, 40_000, 100, 0, "mh_kernel<3,0,0,128,short>"), ("smt", 6, 40_000, 100, 0, "mh_kernel<3,0,0,128>"),
    ("smt", 7, 155_000, 100, 1, "mh_kernel<3,0,0,256>"), ("smt", 2, 155_000, 100, 1, "mh_kernel<3,0,0,256,short>"),
]


@pytest.mark.parametrize("model,k,n,thin,every,kernel", ROUTES)
def test_routes(fake, model, k, n, thin, every, kernel):
    _, gpu = fake
    w = {"monoexp": W.MONOEXP_4K, "mwi3": W.MWI3_1M, "smt": W.SMT_1P5M}[model]
    if k != len(w.acq):
        w = w.with_(acq=tuple(2.0 + 0.7 * np.arange(k)))
    gpu.reset()
    _sampler(fake, w, n, 1, iterations=200, burnin=0, thin=thin, moments_mode=every)
    assert gpu.names() == [kernel]


def test_tiles_reach_every_sm(fake):
    """Full blocks that are too few for the SMs shrink to whole warps of chains."""
    _, gpu = fake
    for n in (20_000, 24_000, 33_000, 38_000, 60_000):
        for prec in (0, 1):
            gpu.reset()
            _sampler(fake, W.MONOEXP_4K, n, 1, iterations=20, burnin=0, thin=5, precision=prec, lanes_per_chain=1)
            assert gpu.launches[0][1] >= 152


@pytest.mark.parametrize("n_acq,per_sm", [(6, 8), (24, 8), (48, 4), (64, 3)])
def test_forward_rows_are_one_wave(fake, n_acq, per_sm):
    _, gpu = fake
    gpu.reset()
    _forward(fake, n_acq, 300_000)
    assert gpu.launches[-1][:2] == ("forward_f_kernel<2>", 152 * per_sm)
    gpu.reset()
    _forward(fake, n_acq, 129)
    assert gpu.launches[-1][1] == 2
