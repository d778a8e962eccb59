"""The exchange protocol of the tile-resident sweeps (csrc/tile.cu) with tiles that
progress at different rates, emulated on the CPU.  A launch reads its halo of the
initial labels from the plane that it writes back to when the number of sweeps is
even (Gibbs: always), so a tile must not write back before its neighbours have
staged; runs of at most one exchange's sweeps therefore make one exchange more.
Tiles are generators: each stages, sweeps, publishes (label, tag) words into one of
two buffers in turn, polls its halo (a wait yields), and writes back.  Whatever the
order, the labels equal the plain sweeps', also over launches that share the
buffers; without the additional exchange some order reads a neighbour's results."""
import numpy as np
import pytest

from test_tile_resident import offsets, plain, toy


def tile(planes, src, dst, g, xch, nb, gibbs, t0, n, k, box, extra):
    """One tile's launch over rows [r0, r1), columns [c0, c1); yields while it waits
    and once before it stages."""
    H, W = g.shape
    r0, r1, c0, c1 = box
    ncol = (2 if nb == 4 else 4) if gibbs else 1
    h = k * ncol
    yield
    near = [(r, c) for r in range(max(r0 - h, 0), min(r1 + h, H))
            for c in range(max(c0 - h, 0), min(c1 + h, W))]
    X = {p: planes[src][p] for p in near}
    own = [(r, c) for r in range(r0, r1) for c in range(c0, c1)]
    halo = [p for p in near if not (r0 <= p[0] < r1 and c0 <= p[1] < c1)]
    if nb == 4 and not gibbs and h == 1:   # no diagonal neighbours are read
        halo = [p for p in halo if r0 <= p[0] < r1 or c0 <= p[1] < c1]
    done, x = 0, 1
    while True:
        ns = min(k, n - done)
        for s in range(ns):
            Y = X if gibbs else dict(X)
            for q in range(ncol):
                e = (ns - s) * ncol - 1 - q
                old = dict(X) if gibbs else X
                for r in range(max(r0 - e, 0), min(r1 + e, H)):
                    for c in range(max(c0 - e, 0), min(c1 + e, W)):
                        col = ((r + c) % 2 if nb == 4 else 2 * (r % 2) + c % 2) if gibbs else 0
                        if col == q:
                            v = [old[r + a, c + b] if 0 <= r + a < H and 0 <= c + b < W else 16
                                 for a, b in offsets(nb)]
                            Y[r, c] = toy(v, old[r, c], g[r, c], t0 + done + s, r, c)
            X = Y
        done += ns
        more = done < n or (extra and x == 1 and src == dst)
        if not more:
            break
        tag, buf = t0 + done, xch[x & 1]
        for r, c in own:
            if r < r0 + h or r >= r1 - h or c < c0 + h or c >= c1 - h:
                buf[r, c] = (X[r, c], tag)
        for p in halo:
            while buf[p][1] != tag:
                assert buf[p][1] < tag   # a neighbour ran two exchanges ahead
                yield
            X[p] = buf[p][0]
        if done == n:
            break
        x += 1
    for p in own:
        planes[dst][p] = X[p]


def launch(planes, src, dst, g, xch, nb, gibbs, t0, n, k, th, tw, order, extra=True):
    H, W = g.shape
    boxes = [(r, min(r + th, H), c, min(c + tw, W)) for r in range(0, H, th) for c in range(0, W, tw)]
    live = {i: tile(planes, src, dst, g, xch, nb, gibbs, t0, n, k, b, extra)
            for i, b in enumerate(boxes)}
    idle = 0
    while live:
        ids = sorted(live)
        if order == "last":
            ids.reverse()
        elif order != "first":
            order.shuffle(ids)
        moved = False
        for i in ids:
            before = sum(v[1] for v in xch[0].flat) + sum(v[1] for v in xch[1].flat)
            steps = 0
            while steps < 3:   # until it blocks: two yields in a row without progress
                try:
                    next(live[i])
                except StopIteration:
                    del live[i]
                    moved = True
                    break
                steps += 1
            moved |= before != sum(v[1] for v in xch[0].flat) + sum(v[1] for v in xch[1].flat)
            if not isinstance(order, str) and order.random() < 0.5:
                break              # another tile's turn
        idle = 0 if moved else idle + 1
        assert idle < 200, "every tile waits"


def run(g, nb, gibbs, runs, k, th, tw, order, extra=True):
    H, W = g.shape
    planes = [g.copy(), np.full_like(g, 99)]
    xch = [np.empty((H, W), object) for _ in range(2)]
    for b in xch:
        for p in np.ndindex(H, W):
            b[p] = (0, 0)
    cur = t0 = 0
    for n in runs:
        dst = cur if gibbs or n % 2 == 0 else cur ^ 1
        launch(planes, cur, dst, g, xch, nb, gibbs, t0, n, k, th, tw, order, extra)
        cur, t0 = dst, t0 + n
    return planes[cur]


def orders():
    rng = np.random.default_rng(5)
    return ["first", "last"] + [np.random.default_rng(s) for s in rng.integers(0, 1000, 3)]


@pytest.mark.parametrize("nb,gibbs", [(4, False), (8, False), (4, True), (8, True)])
@pytest.mark.parametrize("k", [1, 2])
@pytest.mark.parametrize("runs", [(1,), (2,), (4,), (2, 1, 2), (3, 4), (5, 2)])
def test_any_order_of_tiles_gives_the_plain_sweeps(nb, gibbs, k, runs):
    h = k * ((2 if nb == 4 else 4) if gibbs else 1)
    H, W = 2 * h + 3, 2 * h + 4        # 2 to 3 tiles a side, the last ones short
    g = np.random.default_rng(H).integers(0, 15, (H, W))
    want = plain(g, nb, gibbs, sum(runs))
    for order in orders():
        assert (run(g, nb, gibbs, runs, k, h, max(h, 2), order) == want).all()


def test_the_additional_exchange_is_needed():
    for nb, gibbs, n in ((4, False, 2), (8, False, 2), (4, True, 1), (8, True, 1)):
        h = 2 * ((2 if nb == 4 else 4) if gibbs else 1)
        g = np.random.default_rng(7).integers(0, 15, (2 * h + 3, 2 * h + 4))
        want = plain(g, nb, gibbs, n)
        assert any((run(g, nb, gibbs, (n,), 2, h, h, o, extra=False) != want).any()
                   for o in orders())
