"""The server's HBM budget bounds all the device memory of its requests, the
tile-resident sweeps' prefix tables and border exchange included, and admits
what it admitted when slots held no such memory."""
import ctypes

import numpy as np
import pytest

from pcad_inputs import Model, gaussian_noise, greyscale_scene

pytestmark = pytest.mark.gpu

M16 = Model(L=16, pair=1, pair_coef=0.6, pair_T=3, sigma=1.2, inertia=1.0)
M64 = Model(L=64, pair=1, pair_coef=0.2, pair_T=8, sigma=5.0, inertia=2.0)


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


def _pool_used():
    """Bytes in use of the device's default stream-ordered pool."""
    cu = ctypes.CDLL("libcuda.so.1")
    pool, dev, used = ctypes.c_void_p(), ctypes.c_int(), ctypes.c_uint64()
    assert cu.cuCtxGetDevice(ctypes.byref(dev)) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(pool), dev) == 0
    USED_MEM_CURRENT = 7
    assert cu.cuMemPoolGetAttribute(pool, USED_MEM_CURRENT, ctypes.byref(used)) == 0
    return used.value


def _g(m, H, W, seed=4):
    return gaussian_noise(seed + 1, greyscale_scene(seed, H, W, m.L, n_shapes=6), m.sigma, m.L)


def _block(m, H, W):
    """A lower bound of a slot's own block: three label planes and the sums."""
    pitch = (W + 15) // 16 * 16
    return 3 * pitch * H + 4 * H * W


def _alone(pc, g, m, seed, n):
    with pc.Chain(g, m, seed=seed, burn_in=2) as ch:
        ch.run(n)
        return ch.sample(), ch.mean()


def _drain(pc, sv, ids, shapes):
    out = {}
    while len(out) < len(ids):
        pc.pcad_server_step(sv, 16)
        for rid in ids:
            if rid not in out:
                st, s, mean = pc.pcad_server_poll(sv, rid, *shapes[rid])
                if st == 2:
                    out[rid] = (s, mean)
    return out


@pytest.mark.parametrize("m,H,W", [(M16, 400, 401), (M64, 256, 203)], ids=["L16", "L64"])
@pytest.mark.parametrize("policy", [0, 1], ids=["fifo", "srpt"])
# budget in blocks of a request: the block alone, with half an exchange, with
# all of it, and one of the requests' exchanges
@pytest.mark.parametrize("n,spare", [(1, 0.05), (1, 0.3), (1, 0.9), (3, 0.3), (3, 0.9), (3, 3.0)])
def test_budget_bounds_the_slots_memory(pc, m, H, W, policy, n, spare):
    g = _g(m, H, W)
    budget = int((n + spare) * _block(m, H, W) + n * 32768)   # 32 KB: model tables
    sv = pc.pcad_server_create(8, budget)
    try:
        pc.pcad_server_set_policy(sv, policy, 0.2)
        ids = [pc.pcad_server_submit(sv, g, m, 7 + k, 0, 2, 40) for k in range(n)]
        before = _pool_used()
        act, pend, _ = pc.pcad_server_step(sv, 4)
        assert (act, pend) == (n, 0)     # as many as fit without side memory
        held = _pool_used() - before
        used = pc.pcad_server_info(sv)["hbm_used"]
        # beside the slots: work lists and the launches' own small tables
        assert used <= budget
        assert held <= budget + (256 << 10)
        assert abs(held - used) <= (256 << 10)
        res = _drain(pc, sv, ids, {r: g.shape for r in ids})
        assert pc.pcad_server_info(sv)["hbm_used"] == 0
    finally:
        pc.pcad_server_destroy(sv)
    for k, rid in enumerate(ids):
        x, mean = _alone(pc, g, m, 7 + k, 40)
        assert np.array_equal(res[rid][0], x) and np.array_equal(res[rid][1], mean)


@pytest.mark.parametrize("policy", [0, 1], ids=["fifo", "srpt"])
def test_side_memory_makes_room_for_the_next_request(pc, policy):
    """Requests that arrive while others run with side memory are admitted as
    soon as the blocks fit; the others go on without it, with the same results."""
    m, H, W = M64, 256, 203
    g = _g(m, H, W)
    budget = int(3.1 * _block(m, H, W)) + 3 * 32768
    sv = pc.pcad_server_create(8, budget)
    try:
        pc.pcad_server_set_policy(sv, policy, 0.2)
        ids = []
        for k in range(3):
            ids.append(pc.pcad_server_submit(sv, g, m, 7 + k, 0, 2, 60))
            act, pend, _ = pc.pcad_server_step(sv, 7)
            assert (act, pend) == (k + 1, 0)
            assert pc.pcad_server_info(sv)["hbm_used"] <= budget
        res = _drain(pc, sv, ids, {r: g.shape for r in ids})
    finally:
        pc.pcad_server_destroy(sv)
    for k, rid in enumerate(ids):
        x, mean = _alone(pc, g, m, 7 + k, 60)
        assert np.array_equal(res[rid][0], x) and np.array_equal(res[rid][1], mean)


def test_models_that_never_run_tile_resident_hold_no_exchange(pc):
    """c < 0, 8 neighbours with many labels: slots hold their block only."""
    for m in (Model(L=16, pair=1, pair_coef=-0.3, pair_T=3, sigma=1.2, inertia=1.0),
              Model(L=64, nbhd=8, pair=1, pair_coef=0.1, pair_T=8, sigma=5.0, inertia=2.0)):
        g = _g(m, 300, 301)
        sv = pc.pcad_server_create(2, 1 << 30)
        try:
            rid = pc.pcad_server_submit(sv, g, m, 7, 0, 2, 8)
            before = _pool_used()
            pc.pcad_server_step(sv, 4)
            held = _pool_used() - before
            assert held <= _block(m, 300, 301) + (256 << 10)
            _drain(pc, sv, [rid], {rid: g.shape})
        finally:
            pc.pcad_server_destroy(sv)
