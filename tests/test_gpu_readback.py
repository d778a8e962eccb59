"""Read-back of labels: linear copies, packed where the device rows have gaps,
row copies where the host rows do."""
import ctypes

import numpy as np
import pytest

from pcad_inputs import Model

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


@pytest.mark.parametrize("H,W", [(1, 1), (5, 16), (7, 33), (64, 48), (3, 1021)])
def test_labels_read_back_whole(pc, H, W):
    rng = np.random.default_rng(W)
    L = 5
    g = rng.integers(0, L, (H, W)).astype(np.uint8)
    m = Model(L=L, pair=1, pair_coef=0.5, pair_T=2, sigma=1.0, inertia=1.0)
    u8p = ctypes.POINTER(ctypes.c_uint8)
    with pc.Chain(g, m, seed=3, burn_in=0) as ch:
        assert np.array_equal(ch.sample(), g)
        x = rng.integers(0, L, (H, W)).astype(np.uint8)
        ch.set_sample(x)
        assert np.array_equal(ch.sample(), x)
        wide = np.full((H, W + 7), 99, np.uint8)   # host rows with gaps
        assert pc.lib().pcad_chain_read_sample(ch.h, wide.ctypes.data_as(u8p), W + 7) == 0
        assert np.array_equal(wide[:, :W], x) and (wide[:, W:] == 99).all()
        with pc.Chain.from_blob(ch.export()) as c2:
            assert np.array_equal(c2.sample(), x)
        ch.track_energy(4)
        ch.run(2)
        xb, _, sweep = ch.min_state()
        assert xb.max() < L and sweep in (1, 2)
    b = pc.pcad_batch_create([(g, m, 3, 0, 0)], autotune=False)
    try:
        assert np.array_equal(pc.pcad_batch_read_sample(b, 0, H, W), g)
    finally:
        pc.pcad_batch_destroy(b)
