"""The one-launch energy reduction (4 sites per word, ticketed last block)
against the oracle's sums at its edges: words with 1 to 4 sites, one row, one
column, one pixel, and an image of several words per thread; and the tracked
minimum, whose state alternates between two planes, against the trace."""
import numpy as np
import pytest

from oracle import energy as oen
from pcad_inputs import Model, random_lattice

pytestmark = pytest.mark.gpu

MODELS = [Model(L=16, pair=1, pair_coef=0.6, pair_T=3, sigma=1.2, inertia=1.0),
          Model(L=16, nbhd=8, pair=1, pair_coef=0.15, pair_T=30, sigma=1.2, inertia=1.0),
          Model(L=2, nbhd=8, pair=0, pair_coef=0.5, noise=1, flip_p=0.2, inertia=0.5),
          # sweeps that reduce the energy of the state they read
          Model(L=16, nbhd=8, pair=0, pair_coef=0.5, sigma=1.2, inertia=1.0, inertia_norm=1),
          Model(L=20, pair=1, pair_coef=0.2, pair_T=9, sigma=2.0, inertia=1.0, inertia_norm=2)]


@pytest.mark.parametrize("H,W", [(1, 1), (1, 5), (5, 1), (3, 4), (4, 7), (33, 66), (1100, 1031)])
@pytest.mark.parametrize("k", range(len(MODELS)))
def test_sums_and_minimum(H, W, k):
    import paper_2507_14869_gb300 as pc
    m = MODELS[k]
    g = random_lattice(H + W, H, W, m.L)
    with pc.Chain(g, m, seed=2, chain_id=4, burn_in=0) as ch:
        ch.track_energy(16)
        ch.run(12)
        trace, x = ch.energies(), ch.sample()
        xmin, emin, smin = ch.min_state()
        e, pair, data = ch.energy()
        ch.reset()
        steps = []
        for _ in range(12):      # one sweep per call: each state's energy on its own
            ch.run(1)
            steps.append(ch.energy()[0])
    assert np.array_equal(trace, steps)
    assert (pair, data) == oen.energy_terms(m, g, x)
    assert trace[-1] == e
    assert smin == int(np.argmin(trace)) + 1 and emin == trace.min()
    assert oen.posterior_energy(m, g, xmin) == pytest.approx(emin, rel=1e-12, abs=1e-9)
