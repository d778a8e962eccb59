"""Small two-label chains in bands of a cluster of 8 CTAs (halos of 4 rows pushed
through distributed shared memory) against the per-sweep kernel, label for
label: heights whose last bands are short or empty, ragged widths, one and two
quads per thread, and runs of 1 to 9 sweeps (a whole number of exchanges, one
more and one less) of both samplers and neighbourhoods."""
import numpy as np
import pytest

from pcad_inputs import Model, random_lattice

pytestmark = pytest.mark.gpu

RESIDENT, CUDA_CORE = 5, 1


@pytest.mark.parametrize("H,W", [(29, 73), (32, 64), (33, 64), (32, 510), (57, 37), (64, 64),
                                 (100, 160), (513, 4)])
@pytest.mark.parametrize("nbhd", [4, 8])
@pytest.mark.parametrize("sampler", [0, 1], ids=["pca", "gibbs"])
def test_cluster_bands_match(H, W, nbhd, sampler):
    import paper_2507_14869_gb300 as pc
    g = random_lattice(H, H, W, 2)
    m = Model(L=2, nbhd=nbhd, pair=0, pair_coef=0.7, noise=1, flip_p=0.2, inertia=0.6)
    outs = []
    for kind in (RESIDENT, CUDA_CORE):
        with pc.Chain(g, m, seed=9, chain_id=1, burn_in=2, sampler=sampler) as ch:
            ch.set_kernel(kind)
            for n in (1, 4, 5, 3, 2, 8, 9, 7):
                ch.run(n)
            outs.append((ch.sample(), ch.mean(), ch.fp64_draws()))
    assert np.array_equal(outs[0][0], outs[1][0])
    assert np.array_equal(outs[0][1], outs[1][1])
    assert outs[0][2] == outs[1][2]
