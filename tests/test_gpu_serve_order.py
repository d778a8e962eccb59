"""Shortest remaining work first, by the rates of the kernels that run: the request
whose own run takes the GPU less time finishes first."""
import time

import pytest

from pcad_inputs import Model, gaussian_noise, greyscale_scene

pytestmark = pytest.mark.gpu

L16 = Model(L=16, pair=1, pair_coef=0.6, pair_T=3, sigma=1.2, inertia=1.0)
L256 = Model(L=256, pair=1, pair_coef=0.05, pair_T=30, sigma=20.0, inertia=2.0)


def _g(m, side):
    return gaussian_noise(5, greyscale_scene(4, side, side, m.L, n_shapes=6), m.sigma, m.L)


# (model, sweeps) of the longer and of the shorter request, one image size
@pytest.mark.parametrize("slow,fast", [((L16, 800), (L256, 200))], ids=["L16_L256"])
def test_the_shorter_request_finishes_first(slow, fast):
    import paper_2507_14869_gb300 as pc
    side = 400
    alone, order = [], []
    for m, n in (slow, fast):
        with pc.Chain(_g(m, side), m, seed=3, burn_in=0) as ch:
            ch.run(64)
            ch.sync()
            best = 1e9
            for _ in range(3):
                t0 = time.perf_counter()
                ch.run(n)
                ch.sync()
                best = min(best, time.perf_counter() - t0)
            alone.append(best)
    assert alone[1] < 0.9 * alone[0], "the case does not say which one is shorter"
    sv = pc.pcad_server_create(4, 1 << 30)
    try:
        pc.pcad_server_set_policy(sv, pc.SERVE_SRPT, 0.0)   # no aging
        pc.pcad_server_set_limits(sv, 1)                    # one request at a time
        ids = [pc.pcad_server_submit(sv, _g(m, side), m, 3, 0, 0, n) for m, n in (slow, fast)]
        while len(order) < 2:
            pc.pcad_server_step(sv, 16)
            for rid in ids:
                if rid not in order and pc.pcad_server_poll(sv, rid, side, side)[0] == 2:
                    order.append(rid)
    finally:
        pc.pcad_server_destroy(sv)
    assert order == [ids[1], ids[0]]
