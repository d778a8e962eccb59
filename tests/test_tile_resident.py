"""The tile-resident sweeps (csrc/tile.cu) emulated on the CPU: tile geometry,
staged words, the sites of each colour phase, border words published and halo
words polled, on a toy update in place of the draw.  Every word a tile polls
must have been published with the polled sweep's tag (no wait can run out),
every staged index must lie in its plane, and the labels must equal those of
the plain sweep."""
import numpy as np
import pytest

THREADS, MAX_SITES = 512, 8192


def geometry(H, W, ctas, h):
    """tile_geometry of csrc/tile.cu: (th, twq, tiles_x, tiles_y) or None."""
    Wq, best = (W + 3) // 4, None
    for nx in range(1, min(ctas, Wq) + 1):
        twq = -(-Wq // nx)
        tx = -(-Wq // twq)
        th = max(h, -(-H // (ctas // tx)))
        ty = -(-H // th)
        if th * twq * 4 > MAX_SITES or tx * ty > ctas:
            continue
        cost = -(-th * twq * 4 // THREADS) * 1000 + 2 * (th + twq)
        if best is None or cost < best[0]:
            best = (cost, th, twq, tx, ty)
    return best and best[1:]


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


def tiled(g, nb, gibbs, sweeps, ctas):
    H, W = g.shape
    Wq = (W + 3) // 4
    h = 1 if not gibbs else (2 if nb == 4 else 4)
    ncol = 2 if nb == 4 else 4
    TH, TWq, tx_n, ty_n = geometry(H, W, ctas, h)
    TW, SW, SR = 4 * TWq, TWq + 2, TH + 2 * h
    assert tx_n * ty_n <= ctas and tx_n * TWq >= Wq and ty_n * TH >= H and TH >= h
    tiles = []
    for b in range(tx_n * ty_n):
        ty, tx = divmod(b, tx_n)
        r0, c0 = ty * TH, 4 * tx * TWq
        X = np.full((SR, 4 * SW), 16)
        G = np.zeros((SR, 4 * SW), int)
        for sr in range(SR):
            for sb in range(4 * SW):
                r, c = r0 - h + sr, c0 - 4 + sb
                if 0 <= r < H and 0 <= c < W:
                    X[sr, sb], G[sr, sb] = g[r, c], g[r, c]
        tiles.append([r0, c0, X, G])
    out = np.full((H, W), -1)
    xch = np.zeros((2, H, Wq, 5), int)   # 4 labels, tag
    for k in range(sweeps):
        for tile in tiles:
            r0, c0, X, G = tile

            def draw(src, lr, lc):
                sr, sb = lr + h, lc + 4
                n = []
                for a, b in offsets(nb):
                    assert 0 <= sr + a < SR and 0 <= sb + b < 4 * SW
                    n.append(src[sr + a, sb + b])
                return toy(n, src[sr, sb], G[sr, sb], k, r0 + lr, c0 + lc)
            if not gibbs:
                Y = X.copy()   # (the other plane: halo words not polled stay stale there)
                Y[:h], Y[h + TH:], Y[h:h + TH, :4], Y[h:h + TH, 4 + TW:] = 99, 99, 99, 99
                for sr in range(SR):   # outside the image both planes hold 16
                    for sb in range(4 * SW):
                        if not (0 <= r0 - h + sr < H and 0 <= c0 - 4 + sb < W):
                            Y[sr, sb] = 16
                for i in range(TH * TW):
                    lr, lc = divmod(i, TW)
                    assert (i * (0xFFFFFFFF // TW + 1)) >> 32 == lr
                    if r0 + lr < H and c0 + lc < W:
                        Y[lr + h, lc + 4] = draw(X, lr, lc)
                tile[2] = Y
            else:
                for q in range(ncol):
                    e = ncol - 1 - q
                    if nb == 4:
                        nr, per, sr0, sc0 = TH + 2 * e, (TW + 2 * e + 1) >> 1, -e, -e
                    else:
                        sr0 = -e + ((r0 - e + (q >> 1)) & 1)
                        sc0 = -e + ((-e + q) & 1)
                        nr, per = (TH + e - sr0 + 1) >> 1, (TW + e - sc0 + 1) >> 1
                    seen, inv = set(), 0xFFFFFFFF // per + 1
                    for i in range(nr * per):
                        ir = (i * inv) >> 32
                        ic = i - ir * per
                        assert (ir, ic) == divmod(i, per)
                        lr = sr0 + ir if nb == 4 else sr0 + 2 * ir
                        lc = sc0 + 2 * ic
                        if nb == 4:
                            lc += (r0 + lr + c0 + lc + q) & 1
                        if lc < TW + e and 0 <= r0 + lr < H and 0 <= c0 + lc < W:
                            seen.add((lr, lc))
                            X[lr + h, lc + 4] = draw(X, lr, lc)
                    want = {(lr, lc) for lr in range(-e, TH + e) for lc in range(-e, TW + e)
                            if 0 <= r0 + lr < H and 0 <= c0 + lc < W and
                            ((r0 + lr + c0 + lc) % 2 if nb == 4 else
                             2 * ((r0 + lr) % 2) + (c0 + lc) % 2) == q}
                    assert seen == want
        if k + 1 == sweeps:
            break
        buf = xch[(k + 1) & 1]
        for r0, c0, X, _ in tiles:   # publish
            for lr in range(TH):
                for lq in range(TWq):
                    r, q = r0 + lr, c0 // 4 + lq
                    if (lr < h or lr >= TH - h or lq in (0, TWq - 1)) and r < H and q < Wq:
                        buf[r, q, :4] = X[lr + h, 4 * (lq + 1):4 * (lq + 2)]
                        buf[r, q, 4] = k + 1
        for r0, c0, X, _ in tiles:   # poll
            nrow = 2 * h * SW
            for i in range(nrow + 2 * TH):
                if i < nrow:
                    sr, sq = divmod(i, SW)
                    if nb == 4 and not gibbs and sq in (0, SW - 1):
                        continue
                    sr = sr if sr < h else sr + TH
                else:
                    sr, sq = h + ((i - nrow) >> 1), (SW - 1 if i & 1 else 0)
                r, q = r0 - h + sr, c0 // 4 - 1 + sq
                if 0 <= r < H and 0 <= q < Wq:
                    assert buf[r, q, 4] == k + 1   # published this sweep
                    X[sr, 4 * sq:4 * sq + 4] = buf[r, q, :4]
    for r0, c0, X, _ in tiles:
        for lr in range(TH):
            for lc in range(TW):
                if r0 + lr < H and c0 + lc < W:
                    out[r0 + lr, c0 + lc] = X[lr + h, lc + 4]
    return out


@pytest.mark.parametrize("H,W,ctas", [(1, 1, 4), (3, 21, 6), (9, 4, 3), (17, 23, 12), (13, 30, 7),
                                      (26, 11, 9)])
@pytest.mark.parametrize("nb,gibbs", [(4, False), (8, False), (4, True), (8, True)])
def test_tiles_equal_the_plain_sweep(H, W, ctas, nb, gibbs):
    g = np.random.default_rng(H * 100 + W).integers(0, 15, (H, W))
    assert (tiled(g, nb, gibbs, 4, ctas) == plain(g, nb, gibbs, 4)).all()


def test_geometry_fits_the_tiles():
    rng = np.random.default_rng(3)
    for _ in range(300):
        H, W, h = int(rng.integers(1, 1300)), int(rng.integers(1, 1300)), int(rng.choice([1, 2, 4]))
        for ctas in (152, 304):
            t = geometry(H, W, ctas, h)
            if t is None:
                assert H * W > ctas * MAX_SITES // 4
                continue
            th, twq, tx, ty = t
            assert tx * ty <= ctas and th >= h and th * ty >= H and 4 * twq * tx >= W
            assert th * (ty - 1) < H and 4 * twq * (tx - 1) < W   # no empty tile row or column
