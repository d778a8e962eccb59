"""Tile-resident sweeps (mid-size images, whole runs in one cooperative launch)
against the general kernel and the oracle: every draw (small labels, segments,
two labels), lazy PCA and checkerboard Gibbs, both neighbourhoods, widths that
are not multiples of 4, tiles of one row, runs of one, an even and an odd
number of sweeps; and a border word that never arrives."""
import time

import numpy as np
import pytest

import oracle
from pcad_inputs import Model, flip_noise, gaussian_noise, greyscale_scene, shapes_binary

pytestmark = pytest.mark.gpu

CUDA_CORE, POTTS, TL = 1, 0, 1


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


def _img(m, H, W):
    if m.L == 2:
        return flip_noise(5, shapes_binary(4, H, W, 6), 0.1)
    return gaussian_noise(5, greyscale_scene(4, H, W, m.L, n_shapes=6), m.sigma, m.L)


MODELS = {
    "L16": Model(L=16, pair=TL, pair_coef=0.85, pair_T=2, sigma=1.2, inertia=2.0),
    "L5_8nb": Model(L=5, nbhd=8, pair=POTTS, pair_coef=0.9, sigma=1.0, inertia=0.5),
    "L8": Model(L=8, pair=TL, pair_coef=0.3, pair_T=7, sigma=1.0, inertia=0.0),
    "L9_8nb": Model(L=9, nbhd=8, pair=POTTS, pair_coef=1.0, sigma=1.6, inertia=0.7),
    "L2": Model(L=2, pair=POTTS, pair_coef=1.2, noise=1, flip_p=0.1, inertia=1.0),
    "L2_8nb": Model(L=2, nbhd=8, pair=POTTS, pair_coef=0.6, noise=1, flip_p=0.1, inertia=1.0),
    "L24": Model(L=24, pair=TL, pair_coef=0.5, pair_T=3, sigma=2.0, inertia=1.0),
    "L64": Model(L=64, pair=TL, pair_coef=0.2, pair_T=8, sigma=5.0, inertia=2.0),
}


# one row, one column, ragged, more columns than rows, tiles of several rounds
@pytest.mark.parametrize("H,W", [(1, 301), (300, 1), (131, 130), (97, 203), (257, 421)])
@pytest.mark.parametrize("name", list(MODELS))
@pytest.mark.parametrize("sampler", [0, 1], ids=["pca", "gibbs"])
def test_tile_resident_matches(pc, name, H, W, sampler):
    m = MODELS[name]
    g = _img(m, H, W)
    outs = {}
    for kind in (0, CUDA_CORE):
        with pc.Chain(g, m, seed=21, chain_id=2, burn_in=3, sampler=sampler) as ch:
            ch.set_kernel(kind)
            for n in (1, 2, 1, 5):
                ch.run(n)
            x9 = ch.sample()
            ch.run(4)
            ch.sync()
            outs[kind] = (x9, ch.sample(), ch.mean())
            ch.reset()
            ch.run(9)      # the sweep index starts again
            assert np.array_equal(ch.sample(), x9)
    for a, b in zip(outs[0], outs[CUDA_CORE]):
        assert np.array_equal(a, b)
    kw = {} if sampler == 0 else {"order": oracle.ORDER_COLOUR}
    xo, acc, nacc, _ = oracle.run_chain(m, g, 13, 3, seed=21, chain=2, sampler=sampler, **kw)
    assert np.array_equal(outs[0][1], xo)
    assert np.allclose(outs[0][2], acc / nacc, rtol=1e-6, atol=0.0)


@pytest.mark.parametrize("side", [1023, 1024, 1027])
def test_largest_tiles(pc, side):
    """The largest image of the tile-resident rule and its neighbours."""
    m = MODELS["L16"]
    g = _img(m, side, 1024)
    outs = []
    for kind in (0, CUDA_CORE):
        with pc.Chain(g, m, seed=3, burn_in=0) as ch:
            ch.set_kernel(kind)
            ch.run(5)
            ch.sync()
            outs.append((ch.sample(), ch.mean()))
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])


def test_coefficients_change_between_runs(pc):
    """set_model within and out of the draw's models (c < 0), and back."""
    m = MODELS["L9_8nb"]
    g = _img(m, 90, 101)
    ms = [m, Model(**{**m.as_dict(), "pair_coef": -0.4}), Model(**{**m.as_dict(), "pair_coef": 0.5})]
    outs = []
    for kind in (0, CUDA_CORE):
        with pc.Chain(g, m, seed=3, burn_in=2) as ch:
            ch.set_kernel(kind)
            ch.run_schedule(ms, [5, 6, 7])
            ch.sync()
            outs.append((ch.sample(), ch.mean()))
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("sampler", [0, 1], ids=["pca", "gibbs"])
def test_a_border_word_that_never_arrives(pc, sampler):
    """A tile that never publishes: every wait is bounded, the launch ends and
    reports PCAD_ETIMEOUT, and the chain runs again after a reset."""
    m = MODELS["L9_8nb"]
    g = _img(m, 200, 220)
    with pc.Chain(g, m, seed=3, burn_in=0, sampler=sampler) as ch:
        ch.run(8)
        ch.sync()
        want = ch.sample()
        ch.set_wait_limit(0.005)
        ch.inject_stall(3)
        ch.reset()
        t0 = time.perf_counter()
        ch.run(8)
        with pytest.raises(pc.PcadError) as e:
            ch.sync()
        assert e.value.status == 4 and time.perf_counter() - t0 < 1.0
        ch.inject_stall(-1)
        ch.set_wait_limit(1.0)
        ch.reset()
        ch.run(8)
        ch.sync()
        assert np.array_equal(ch.sample(), want)


def test_batch_packs_and_server_slices(pc):
    """More chains of one kind than a launch holds, several kinds, a model that
    leaves its kind mid-run; the same chains through the server."""
    rng = np.random.default_rng(8)
    jobs = []
    for k, name in enumerate(["L16"] * 36 + ["L64"] * 4 + ["L2"] * 3 + ["L9_8nb"] * 3 + ["L5_8nb"]):
        H, W = int(rng.integers(60, 150)), int(rng.integers(70, 200))
        jobs.append((_img(MODELS[name], H, W), MODELS[name], 50 + k, k, 4))
    neg = Model(**{**MODELS["L16"].as_dict(), "pair_coef": -0.3})
    want = []
    for k, (g, m, seed, chain, burn) in enumerate(jobs):
        with pc.Chain(g, m, seed=seed, chain_id=chain, burn_in=burn) as ch:
            ch.set_kernel(CUDA_CORE)
            ch.run(23)
            x, mu = ch.sample(), ch.mean()
            if k == 5:
                ch.set_model(neg)
            ch.run(10)
            want.append((x, mu, ch.sample(), ch.mean()))
    b = pc.pcad_batch_create(jobs, autotune=False)
    try:
        for rep in range(2):
            if rep:
                pc.pcad_batch_reset(b)
                pc.pcad_batch_set_model(b, 5, jobs[5][1])
            for n in (7, 16):
                pc.pcad_batch_run(b, n)
            pc.pcad_batch_sync(b)
            for k, (g, *_) in enumerate(jobs):
                assert np.array_equal(pc.pcad_batch_read_sample(b, k, *g.shape), want[k][0]), k
                assert np.array_equal(pc.pcad_batch_read_mean(b, k, *g.shape), want[k][1]), k
            pc.pcad_batch_set_model(b, 5, neg)
            pc.pcad_batch_run(b, 10)
            pc.pcad_batch_sync(b)
            for k, (g, *_) in enumerate(jobs):
                assert np.array_equal(pc.pcad_batch_read_sample(b, k, *g.shape), want[k][2]), k
                assert np.array_equal(pc.pcad_batch_read_mean(b, k, *g.shape), want[k][3]), k
    finally:
        pc.pcad_batch_destroy(b)
    sv = pc.pcad_server_create(64, 10 ** 9)
    try:
        ids = {pc.pcad_server_submit(sv, g, m, s, c, bi, 23): k
               for k, (g, m, s, c, bi) in enumerate(jobs)}
        while ids:
            pc.pcad_server_step(sv, 5)
            for rid in list(ids):
                st, x, mu = pc.pcad_server_poll(sv, rid, *jobs[ids[rid]][0].shape)
                if st == 2:
                    k = ids.pop(rid)
                    assert np.array_equal(x, want[k][0]) and np.array_equal(mu, want[k][1]), k
    finally:
        pc.pcad_server_destroy(sv)
