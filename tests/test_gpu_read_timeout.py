"""Reads after a bounded wait gave up.  A user's pass is reset, run, sample,
mean, metrics, with no sync of its own: every call that hands back what the
sweeps left must report PCAD_ETIMEOUT, not the planes of a launch that ended
early.  (A tile that never publishes, with a 5 ms limit, as in
test_gpu_failure.py: no wait is endless.)"""
import numpy as np
import pytest

from pcad_inputs import Model, flip_noise, gaussian_noise, greyscale_scene, shapes_binary

pytestmark = pytest.mark.gpu

ETIMEOUT = 4


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


# name: model, sampler, kernel kind (0: AUTO, tile-resident at this size)
CASES = {
    "tile_L9": (Model(L=9, nbhd=8, pair=0, pair_coef=1.0, sigma=1.6, inertia=0.7), 0, 0),
    "tile_L5_gibbs": (Model(L=5, nbhd=8, pair=0, pair_coef=0.9, sigma=1.0), 1, 0),
    "tile_L64": (Model(L=64, pair=1, pair_coef=0.2, pair_T=8, sigma=5.0, inertia=2.0), 0, 0),
    "tile_L2": (Model(L=2, pair=0, pair_coef=1.2, noise=1, flip_p=0.1, inertia=1.0), 0, 0),
    "wave_L16": (Model(L=16, pair=1, pair_coef=0.6, pair_T=3, sigma=1.0, inertia=1.5), 0, 3),
}

READS = {
    "sample": lambda ch, clean: ch.sample(),
    "mean": lambda ch, clean: ch.mean(),
    "metrics": lambda ch, clean: ch.metrics(clean),
    "metrics_sample": lambda ch, clean: ch.metrics(clean, 1),
    "energy": lambda ch, clean: ch.energy(),
    "export": lambda ch, clean: ch.export(),
    "sync": lambda ch, clean: ch.sync(),
}


@pytest.mark.parametrize("name", list(CASES))
def test_reads_report_a_wait_that_gave_up(pc, name):
    m, sampler, kind = CASES[name]
    H, W = 200, 220
    if m.L == 2:
        clean = shapes_binary(4, H, W, 6)
        g = flip_noise(5, clean, 0.1)
    else:
        clean = greyscale_scene(4, H, W, m.L, n_shapes=6)
        g = gaussian_noise(5, clean, m.sigma, m.L)
    with pc.Chain(g, m, seed=3, burn_in=0, sampler=sampler) as ch:
        ch.set_kernel(kind)
        ch.run(32)
        want = {k: f(ch, clean) for k, f in READS.items()}
        ch.set_wait_limit(0.005).inject_stall(3).reset()
        ch.run(32)
        for _ in range(6):   # (a chain's checks change to a pinned word after 32)
            for k, f in READS.items():
                with pytest.raises(pc.PcadError) as e:
                    f(ch, clean)
                assert e.value.status == ETIMEOUT, k
        # off again: the reset clears the flag and the reads give the run's results
        ch.inject_stall(-1).reset()
        ch.run(32)
        for k, f in READS.items():
            got = f(ch, clean)
            if isinstance(got, np.ndarray):
                assert np.array_equal(got, want[k]), k
            elif k.startswith("metrics"):
                # sums of 4e4 FP64 terms by atomics, in no fixed order: 4e4 2^-53
                assert np.allclose(got, want[k], rtol=1e-11, atol=0.0), k
            elif k != "sync":
                assert got == want[k], k


def test_a_run_before_the_kernel_changed_is_still_reported(pc):
    """The flag belongs to the sweeps that were issued, not to the kernel
    chosen since."""
    m, _, _ = CASES["wave_L16"]
    g = gaussian_noise(5, greyscale_scene(4, 200, 220, m.L, n_shapes=6), m.sigma, m.L)
    with pc.Chain(g, m, seed=3, burn_in=0) as ch:
        ch.set_kernel(3)
        ch.run(32)
        ch.sync()
        ch.set_wait_limit(0.005).inject_stall(3).reset()
        ch.run(32)
        ch.set_kernel(1)
        with pytest.raises(pc.PcadError) as e:
            ch.sync()
        assert e.value.status == ETIMEOUT
