"""The tile-resident sweeps (csrc/tile.cu) emulated on the CPU: staged words,
the sites of each sweep and colour phase, border words published and halo words
polled, several sweeps per exchange, on a toy update in place of the draw.
Every word a tile polls must have been published with the awaited tag (no wait
can run out), every staged index must lie in its plane, every uniform must have
been computed, and the labels must equal those of the plain sweep."""
import numpy as np
import pytest


def geometry(H, W, ctas, k, phases):
    """The tile grids tile_geometry of csrc/tile.cu weighs for k sweeps per
    exchange: (th, twq, tiles_x, tiles_y) each."""
    Wq, h = (W + 3) // 4, k * phases
    hq = (h + 3) // 4
    for nx in range(1, min(ctas, Wq) + 1):
        twq = max(hq, -(-Wq // nx))
        tx = -(-Wq // twq)
        th = max(h, -(-H // (ctas // tx)))
        ty = -(-H // th)
        if th * twq * 4 <= 8192 and tx * ty <= ctas:
            yield th, twq, tx, ty


def toy(n, x, g, t, r, c):
    """A label from the neighbours' labels (16: missing), as the draw's inputs."""
    return int((sum((j + 3) * (v + 1) for j, v in enumerate(n)) + 5 * x + 7 * g + 11 * t +
                13 * r + 17 * c) % 15)


def offsets(nb):
    o = [(-1, 0), (1, 0), (0, -1), (0, 1)]
    return o + [(-1, -1), (-1, 1), (1, -1), (1, 1)] if nb == 8 else o


def plain(g, nb, gibbs, sweeps):
    H, W = g.shape
    x = np.full((H + 2, W + 2), 16)
    x[1:-1, 1:-1] = g
    for t in range(sweeps):
        ncol = (2 if nb == 4 else 4) if gibbs else 1
        for q in range(ncol):
            src = x.copy()
            for r in range(H):
                for c in range(W):
                    col = ((r + c) % 2 if nb == 4 else 2 * (r % 2) + c % 2) if gibbs else 0
                    if col == q:
                        x[r + 1, c + 1] = toy([src[r + 1 + a, c + 1 + b] for a, b in offsets(nb)],
                                              src[r + 1, c + 1], g[r, c], t, r, c)
    return x[1:-1, 1:-1]


def tiled(g, nb, gibbs, sweeps, th, twq, k, words=False):
    H, W = g.shape
    Wq = (W + 3) // 4
    ncol = (2 if nb == 4 else 4) if gibbs else 1
    h = k * ncol
    hq = (h + 3) // 4
    hb, TH, TWq, TW = 4 * hq, th, twq, 4 * twq
    SW, SR = TWq + 2 * hq, TH + 2 * h
    assert TH >= h and TWq >= hq
    tx_n, ty_n = -(-Wq // TWq), -(-H // TH)
    tiles = []
    for b in range(tx_n * ty_n):
        ty, tx = divmod(b, tx_n)
        r0, c0 = ty * TH, 4 * tx * TWq
        X = np.full((SR, 4 * SW), 16)
        G = np.zeros((SR, 4 * SW), int)
        for sr in range(SR):
            for sb in range(4 * SW):
                r, c = r0 - h + sr, c0 - hb + sb
                if 0 <= r < H and 0 <= c < W:
                    X[sr, sb], G[sr, sb] = g[r, c], g[r, c]
        inside = np.array([[0 <= r0 - h + sr < H and 0 <= c0 - hb + sb < W
                            for sb in range(4 * SW)] for sr in range(SR)])
        tiles.append([r0, c0, X, G, inside])
    xch = np.zeros((2, H, Wq, 5), int)   # 4 labels, tag
    done, x = 0, 1
    while True:
        ns = min(k, sweeps - done)
        for tile in tiles:
            r0, c0, X, G, inside = tile
            for s in range(ns):
                # quads whose uniforms sweep s has
                e0 = (ns - s) * ncol - 1
                eq = (e0 + 3) >> 2
                per, U = TWq + 2 * eq, set()
                for i in range((TH + 2 * e0) * per):
                    ir = i if per == 1 else (i * (0xFFFFFFFF // per + 1)) >> 32
                    lr, lq = ir - e0, i - ir * per - eq
                    assert divmod(i, per) == (ir, lq + eq)
                    assert 0 <= lr + h < SR and 0 <= lq + hq < SW
                    U.add((lr, lq))
                # the other plane: stale but outside the image
                Y = X if gibbs else np.where(inside, 99, 16)
                for q in range(ncol):
                    e = (ns - s) * ncol - 1 - q
                    if not gibbs:
                        nr, per, sr0, sc0 = TH + 2 * e, TW + 2 * e, -e, -e
                    elif nb == 4:
                        nr, per, sr0, sc0 = TH + 2 * e, (TW + 2 * e + 1) >> 1, -e, -e
                    else:
                        sr0 = -e + ((r0 - e + (q >> 1)) & 1)
                        sc0 = -e + ((-e + q) & 1)
                        nr, per = (TH + e - sr0 + 1) >> 1, (TW + e - sc0 + 1) >> 1
                    seen, inv = set(), 0xFFFFFFFF // per + 1
                    if words:   # 4 sites of a word at a time; its other sites undefined
                        perw, eqw = TWq + 2 * ((e + 3) >> 2), (e + 3) >> 2
                        for i in range((TH + 2 * e) * perw):
                            ir = i if perw == 1 else (i * (0xFFFFFFFF // perw + 1)) >> 32
                            lr, lq = ir - e, i - ir * perw - eqw
                            lo = max(-e - 4 * lq, 0)
                            hi = min(TW + e - 4 * lq, W - c0 - 4 * lq, 4)
                            if not (0 <= r0 + lr < H and c0 + 4 * lq >= 0 and lo < hi):
                                continue
                            assert (lr, lq) in U
                            o = (lr + h) * SW + lq + hq   # words read around it
                            assert SW <= o and o + SW + 1 <= SR * SW
                            for b in range(4):
                                lc, sr, sb = 4 * lq + b, lr + h, 4 * (lq + hq) + b
                                if not lo <= b < hi:
                                    Y[sr, sb] = 99 if inside[sr, sb] else 16
                                    continue
                                seen.add((lr, lc))
                                n = [X[sr + a, sb + c] for a, c in offsets(nb)]
                                assert 0 < sb < 4 * SW - 1 and 99 not in n
                                Y[sr, sb] = toy(n, X[sr, sb], G[sr, sb], done + s, r0 + lr, c0 + lc)
                    for i in range(0 if words else nr * per):
                        ir = (i * inv) >> 32
                        ic = i - ir * per
                        assert (ir, ic) == divmod(i, per)
                        lr = sr0 + 2 * ir if gibbs and nb == 8 else sr0 + ir
                        lc = sc0 + (2 * ic if gibbs else ic)
                        if gibbs and nb == 4:
                            lc += (r0 + lr + c0 + lc + q) & 1
                        if not (lc < TW + e and 0 <= r0 + lr < H and 0 <= c0 + lc < W):
                            continue
                        seen.add((lr, lc))
                        assert (lr, lc >> 2) in U
                        sr, sb = lr + h, lc + hb
                        n = []
                        for a, b in offsets(nb):
                            assert 0 <= sr + a < SR and 0 <= sb + b < 4 * SW
                            n.append(X[sr + a, sb + b])
                        assert 99 not in n
                        Y[sr, sb] = toy(n, X[sr, sb], G[sr, sb], done + s, r0 + lr, c0 + lc)
                    want = {(lr, lc) for lr in range(-e, TH + e) for lc in range(-e, TW + e)
                            if 0 <= r0 + lr < H and 0 <= c0 + lc < W and
                            (not gibbs or ((r0 + lr + c0 + lc) % 2 if nb == 4 else
                                           2 * ((r0 + lr) % 2) + (c0 + lc) % 2) == q)}
                    assert seen == want
                X = tile[2] = Y
        done += ns
        if done == sweeps:
            break
        buf = xch[x & 1]
        for r0, c0, X, _, _ in tiles:   # publish
            for lr in range(TH):
                for lq in range(TWq):
                    r, q = r0 + lr, c0 // 4 + lq
                    border = lr < h or lr >= TH - h or lq < hq or lq >= TWq - hq
                    if border and r < H and q < Wq:
                        buf[r, q, :4] = X[lr + h, 4 * (lq + hq):4 * (lq + hq + 1)]
                        buf[r, q, 4] = done
        corners = nb == 8 or gibbs or h > 1
        for r0, c0, X, _, _ in tiles:   # poll
            nrow = 2 * h * SW
            for i in range(nrow + 2 * hq * TH):
                if i < nrow:
                    sr, sq = divmod(i, SW)
                    if not corners and (sq < hq or sq >= SW - hq):
                        continue
                    sr = sr if sr < h else sr + TH
                else:
                    sr, sq = divmod(i - nrow, 2 * hq)
                    sr += h
                    sq = sq if sq < hq else sq + TWq
                r, q = r0 - h + sr, c0 // 4 - hq + sq
                if 0 <= r < H and 0 <= q < Wq:
                    assert buf[r, q, 4] == done   # published this exchange
                    X[sr, 4 * sq:4 * sq + 4] = buf[r, q, :4]
        x += 1
    out = np.full((H, W), -1)
    for r0, c0, X, _, _ in tiles:
        for lr in range(TH):
            for lc in range(TW):
                if r0 + lr < H and c0 + lc < W:
                    out[r0 + lr, c0 + lc] = X[lr + h, lc + hb]
    return out


@pytest.mark.parametrize("H,W,th,twq", [(1, 1, 1, 1), (3, 21, 2, 1), (9, 4, 4, 1), (17, 23, 5, 2),
                                        (13, 30, 8, 3), (26, 11, 9, 2), (19, 37, 16, 4)])
@pytest.mark.parametrize("nb,gibbs", [(4, False), (8, False), (4, True), (8, True)])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_tiles_equal_the_plain_sweep(H, W, th, twq, nb, gibbs, k):
    h = k * ((2 if nb == 4 else 4) if gibbs else 1)
    th, twq = max(th, h), max(twq, (h + 3) // 4)
    g = np.random.default_rng(H * 100 + W).integers(0, 15, (H, W))
    want = plain(g, nb, gibbs, 4)
    assert (tiled(g, nb, gibbs, 4, th, twq, k) == want).all()
    if not gibbs:
        assert (tiled(g, nb, gibbs, 4, th, twq, k, words=True) == want).all()


def test_grids_cover_the_image():
    rng = np.random.default_rng(3)
    for _ in range(200):
        H, W = int(rng.integers(1, 1300)), int(rng.integers(1, 1300))
        k, phases, ctas = int(rng.integers(1, 5)), int(rng.choice([1, 2, 4])), int(rng.choice([152, 304]))
        for th, twq, tx, ty in geometry(H, W, ctas, k, phases):
            h = k * phases
            assert tx * ty <= ctas and th >= h and 4 * twq >= h
            assert th * ty >= H and 4 * twq * tx >= W
            assert th * (ty - 1) < H and 4 * twq * (tx - 1) < W   # no empty tile row or column
