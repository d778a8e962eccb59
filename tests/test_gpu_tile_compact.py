"""Compact two-label tiles (images above 8192 sites per tile: uniforms drawn in
the pass, sums as bytes) against the general kernel: ragged sizes, both
neighbourhoods, runs that fill the byte counts (255 sums), and short runs
between them on the per-sweep kernel."""
import numpy as np
import pytest

from pcad_inputs import Model, random_lattice

pytestmark = pytest.mark.gpu

CUDA_CORE = 1


@pytest.mark.parametrize("H,W", [(1597, 1603), (700, 3802), (2901, 1001)])
@pytest.mark.parametrize("nbhd", [4, 8])
def test_compact_tiles_match(H, W, nbhd):
    import paper_2507_14869_gb300 as pc
    g = random_lattice(H, H, W, 2)
    m = Model(L=2, nbhd=nbhd, pair=0, pair_coef=0.7, noise=1, flip_p=0.2, inertia=0.6)
    outs = []
    for kind in (0, CUDA_CORE):
        with pc.Chain(g, m, seed=9, chain_id=1, burn_in=2) as ch:
            ch.set_kernel(kind)
            ch.run(17)
            x = ch.sample()
            for n in (3, 275, 16):
                ch.run(n)
            outs.append((x, ch.sample(), ch.mean(), ch.fp64_draws()))
    assert np.array_equal(outs[0][0], outs[1][0])
    assert np.array_equal(outs[0][1], outs[1][1])
    assert np.array_equal(outs[0][2], outs[1][2])
