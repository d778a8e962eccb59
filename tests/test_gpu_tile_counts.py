"""The FP64 re-draw count of tile-resident runs: sites of a tile's halo are drawn
by several blocks and counted by their owner only, so the count is that of the
same draw with a launch per sweep (runs of one sweep, or the kernel asked for)."""
import numpy as np
import pytest

from pcad_inputs import Model, flip_noise, gaussian_noise, greyscale_scene, shapes_binary

pytestmark = pytest.mark.gpu

CUDA_CORE, WINDOW, BINARY = 1, 6, 8
L2 = Model(L=2, pair=0, pair_coef=1.2, noise=1, flip_p=0.1, inertia=1.0)
L2_8 = Model(L=2, nbhd=8, pair=0, pair_coef=0.6, noise=1, flip_p=0.1, inertia=1.0)
L9_8 = Model(L=9, nbhd=8, pair=0, pair_coef=1.0, sigma=1.6, inertia=0.7)
L16 = Model(L=16, pair=1, pair_coef=0.85, pair_T=2, sigma=1.2, inertia=2.0)
L64 = Model(L=64, pair=1, pair_coef=0.2, pair_T=8, sigma=5.0, inertia=2.0)


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


# model, sampler, image, the per-sweep form: a kernel kind, or None for runs of one sweep
CASES = [
    (L2, 0, 163, 201, BINARY), (L2_8, 0, 163, 201, BINARY), (L2, 0, 601, 803, BINARY),
    (L2, 0, 1403, 1801, BINARY), (L2_8, 1, 163, 201, CUDA_CORE), (L2, 1, 163, 201, CUDA_CORE),
    (L9_8, 0, 97, 203, None), (L9_8, 0, 300, 401, None), (L16, 0, 97, 203, None),
    (L16, 0, 800, 1001, None), (L64, 0, 131, 203, WINDOW), (L64, 0, 300, 301, WINDOW),
    (L64, 1, 131, 203, WINDOW),
]


@pytest.mark.parametrize("m,sampler,H,W,kind", CASES,
                         ids=[f"L{c[0].L}_{c[0].nbhd}nb_{c[1]}_{c[2]}x{c[3]}" for c in CASES])
def test_redraws_are_counted_once(pc, m, sampler, H, W, kind):
    if m.L == 2:
        g = flip_noise(5, shapes_binary(4, H, W, 6), 0.1)
    else:
        g = gaussian_noise(5, greyscale_scene(4, H, W, m.L, n_shapes=6), m.sigma, m.L)
    out = []
    for per_sweep in (False, True):
        with pc.Chain(g, m, seed=21, chain_id=2, burn_in=3, sampler=sampler) as ch:
            if per_sweep and kind is not None:
                ch.set_kernel(kind)
            for n in ([1] * 48 if per_sweep and kind is None else [24, 17, 7]):
                ch.run(n)
            ch.sync()
            out.append((ch.sample(), ch.mean(), ch.fp64_draws()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]
    assert m.L == 2 or out[0][2] > 0     # (two labels: a band may hold no draw)
