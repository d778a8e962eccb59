"""The segment draw (csrc/seg_draw.cuh) replayed in numpy on the CPU: the
exchange network of its 12 kinks, the prefix-table indices, the FP32 segment
sums, the choice and search of the segment and the certified margin, against
the exact FP64 conditional CDF of Eq. posterior_pca_transition_matrix (5.2).

For every site the label that the replay certifies must be the FP64 inverse
CDF's, with uniforms on and around every boundary, ex2 pushed 2 ulp either
way, and every CDF value at a kink must lie within the margin."""
import numpy as np
import pytest

U = 2.0 ** -24
LOG2E = 1.4426950408889634074
f32, f64 = np.float32, np.float64
MISSING = 1024
NET = ([(0, 4), (1, 5), (2, 6), (3, 7), (2, 4), (3, 5), (1, 2), (3, 4), (5, 6)] +
       [(0, 8), (1, 9), (2, 10), (3, 11), (4, 8), (5, 9), (6, 10), (7, 11), (2, 4), (3, 5),
        (6, 8), (7, 9), (1, 2), (3, 4), (5, 6), (7, 8), (9, 10)])


def _fma(a, b, c):   # exact product and sum in FP64 for these magnitudes, one rounding
    return (np.asarray(a, f64) * np.asarray(b, f64) + np.asarray(c, f64)).astype(f32)


def _offset(alpha, mu, L, T):
    """seg_offset of csrc/seg.cu: the scales' offset S, or None."""
    A, rng = mu * 4 * T, L - 1 + T
    S = np.ceil(max(0.0, 4 * mu * rng + A - 125.0))
    sigma = np.sqrt(0.5 * LOG2E / -alpha) if alpha < 0 else 1e9
    if S > 0 and (127.0 - S) / (4 * mu) < min(rng, 5 * sigma + T):
        return None
    d = L - 1.0 if alpha == 0 else min(L - 1.0, 2 * mu / -alpha)
    return S if alpha * d * d + 4 * mu * d - S <= 117.0 else None


def _table(alpha64, mu, L, S):
    """F_k(i) at [k + 4, i + 256]."""
    d = np.arange(-255, 256, dtype=f64)
    out = np.zeros((9, 512))
    for k in range(-4, 5):
        e = np.where(np.abs(d) < L, alpha64 * d * d + float(mu) * k * d - S, -np.inf)
        assert e.max() <= 117.5
        v = np.exp2(e)
        if k >= 0:
            out[k + 4, 1:] = np.cumsum(v)
            out[k + 4] += 2.0 ** -101
        else:
            out[k + 4, :511] = -np.cumsum(v[::-1])[::-1]
            out[k + 4] -= 2.0 ** -101
    t = out.astype(f32)
    t[np.abs(t) < 2.0 ** -126] = 0
    return t


def _sorted_kinks(x, g, T):
    xs = np.sort(8 * (x - g[:, None]), 1)
    k = np.concatenate([xs - 8 * T, xs + 1, xs + 8 * T], 1)
    for a, b in NET:
        lo, hi = np.minimum(k[:, a], k[:, b]), np.maximum(k[:, a], k[:, b])
        k[:, a], k[:, b] = lo, hi
    return k


def _prepare(mod, x, g, xi, ulp):
    """Segment records of every site: Gd, sc, (at, end), G, Z, delta, E1, E2, |v|."""
    L, T = mod["L"], mod["T"]
    lam, c_e, sig = (float(f32(mod[n])) for n in ("inertia", "pair_coef", "sigma"))
    gam = f32(-c_e * LOG2E)
    mu4 = f32(-0.25) * gam
    alpha64 = 0.0 if mod["noise"] == 2 else -LOG2E / (2.0 * sig * sig)
    alpha = f32(alpha64)
    cb = f32(float(gam) * 4 * T)
    S = _offset(float(alpha), -float(gam), L, T)
    assert S is not None
    cbs = f32(f64(cb) + S)
    em1 = f32(np.expm1(lam))
    tab = _table(alpha64, -gam, L, S).reshape(-1)

    def ex2(c):
        with np.errstate(over="ignore"):   # beyond 2^128: an infinity
            e = np.exp2(np.asarray(c, f64)).astype(f32)
        e = (e.astype(f64) * (1.0 + ulp * 2 * U)).astype(f32)
        return np.where(np.asarray(c) < -126.0, f32(0), e)

    n = len(g)
    key = _sorted_kinks(x, g, T)
    assert (np.diff(key, axis=1) >= 0).all()   # the network sorts
    lo, hi = -g, L - g
    Pb = (np.maximum(T - np.abs(xi[:, None] - x), 0)).sum(1)
    iv = _fma(-gam, Pb, cb)
    v = _fma(alpha, (xi - g) ** 2, iv)
    delta = (ex2(v).astype(f64) * f64(em1)).astype(f32) if lam > 0 else np.zeros(n, f32)
    row = np.full(n, 4)
    C = np.zeros(n, np.int64)
    G = np.zeros(n, f32)
    E1, E2 = np.zeros(n, f32), np.zeros(n, f32)
    at = lo + 255 + 512 * row
    p = tab[at]
    s = ex2(np.full(n, cbs))
    s0, c = s, np.zeros(n, f32)
    Gd, sc, ends = [], [], []
    for i in range(13):
        if i < 12:
            pr = np.minimum(key[:, i] >> 3, hi)
            pc = np.maximum(pr, lo)
            dk = 1 - 3 * (key[:, i] & 1)
        else:
            pc = hi
        end = pc + 255 + 512 * row
        assert (row >= 0).all() and (row <= 8).all()
        assert (end >= 0).all() and (end < 9 * 512).all() and (end >= at).all()
        q = tab[end]
        D = q - p
        assert (D >= 0).all()
        w = (D.astype(f64) * s).astype(f32)   # 0 times an infinite scale: NaN, uncertain
        E1 = _fma(np.abs(p) + np.abs(q), s, E1)
        E2 = _fma(w, np.abs(c), E2)
        G = w if i == 0 else G + w
        sc.append(s)
        ends.append((at, end))
        if i == 12:
            break
        Gd.append(np.where(pc > xi - g, G + delta, G))
        row = row + dk
        C = C - dk * pr
        at = pc + 255 + 512 * row
        p = tab[at]
        if i < 11:
            assert (np.abs(4 * C) < 2 ** 22).all()
            c = _fma(mu4, 4 * C, cbs)
            assert (c >= -126.0).all()   # no scale is flushed
            s = ex2(c)
        else:
            c, s = np.zeros(n, f32), s0
    return dict(tab=tab, Gd=Gd, sc=sc, ends=ends, G=G, Z=G + delta, delta=delta, E1=E1, E2=E2,
                av=np.abs(v) + np.abs(iv), cb=cb, kd=6 + f32(0.7) * np.abs(cbs))


def _draw(mod, r, g, xi, ub):
    """(label, certain, margin) per site for the uniform numerators ub."""
    L, tab, n = mod["L"], r["tab"], len(g)
    t = ((ub.astype(f32) * f32(2.0 ** -24)).astype(f64) * r["Z"]).astype(f32)
    Gp, scs = np.zeros(n, f32), r["sc"][0].copy()
    l, h = r["ends"][0][0].copy(), r["ends"][0][1].copy()
    for i in range(12):
        m = t >= r["Gd"][i]
        Gp, scs = np.where(m, r["Gd"][i], Gp), np.where(m, r["sc"][i + 1], scs)
        l, h = np.where(m, r["ends"][i + 1][0], l), np.where(m, r["ends"][i + 1][1], h)
    ax = (l & ~511) + (xi - g) + 256
    f0 = tab[l]
    tt = t - Gp
    xin = (ax > l) & (ax <= h)
    fx = tab[ax - 1]
    cx = (scs.astype(f64) * (fx - f0)).astype(f32)
    tm = tt - r["delta"]
    with np.errstate(all="ignore"):
        y = f0 + tt / scs
        y = np.where(xin & (tt >= cx), np.where(tm > cx, f0 + tm / scs, fx), y)
    lo, hi = l.copy(), h.copy()
    while ((hi - lo) > 1).any():
        mid = (lo + hi) >> 1
        go = (hi - lo) > 1
        up = tab[mid] > y
        hi, lo = np.where(go & up, mid, hi), np.where(go & ~up, mid, lo)
    f1, fl = tab[hi], tab[np.maximum(hi - 1, l)]
    sl = (hi & 511) - 256 + g
    hiC, loC = _fma(scs, f1 - f0, Gp), _fma(scs, fl - f0, Gp)
    hiC = np.where(xin & (hi >= ax), hiC + r["delta"], hiC)
    loC = np.where(xin & (hi > ax), loC + r["delta"], loC)
    M = (f32(1.25 * U) * (r["E1"] + 2 * np.maximum(np.abs(f1), np.abs(fl)) * scs +
                          f32(0.6931472) * (r["E2"] - r["cb"] * r["Z"]) + 22 * r["Z"] +
                          (f32(1.39) * r["av"] + r["kd"]) * r["delta"])).astype(f32)
    certain = (t < hiC) & ((sl == L - 1) | (hiC - t > M)) & ((sl == 0) | (t - loC > M))
    return np.clip(sl, 0, L - 1), certain, M


def _exact_cdf(mod, x, g, xi):
    L, T = mod["L"], mod["T"]
    lam, c_e, sig = (float(f32(mod[n])) for n in ("inertia", "pair_coef", "sigma"))
    s = np.arange(L)
    Pb = np.maximum(T - np.abs(s[None, None, :] - x[:, :, None]), 0).sum(1)
    e = c_e * Pb
    if mod["noise"] != 2:
        e = e - (g[:, None] - s[None, :]) ** 2 / (2.0 * sig * sig)
    e = e + lam * (s[None, :] == xi[:, None])
    w = np.exp(e - e.max(1, keepdims=True))
    return np.cumsum(w, 1)


MODELS = [
    dict(L=256, T=30, pair_coef=0.05, sigma=25.0, inertia=2.0, noise=0),
    dict(L=256, T=30, pair_coef=0.068, sigma=40.0, inertia=0.0, noise=0),
    dict(L=256, T=30, pair_coef=0.08, sigma=39.0, inertia=2.0, noise=0),
    dict(L=256, T=30, pair_coef=0.08, sigma=6.0, inertia=1.0, noise=0),
    dict(L=17, T=2, pair_coef=1.27, sigma=0.4, inertia=2.0, noise=0),
    dict(L=256, T=30, pair_coef=0.03, sigma=5.0, inertia=3.0, noise=0),
    dict(L=256, T=1, pair_coef=0.08, sigma=15.0, inertia=1.5, noise=0),
    dict(L=33, T=4, pair_coef=0.5, sigma=2.6, inertia=1.0, noise=0),
    dict(L=9, T=2, pair_coef=1.6, sigma=0.6, inertia=2.0, noise=0),
    dict(L=100, T=33, pair_coef=0.1, sigma=8.0, inertia=40.0, noise=0),
    dict(L=256, T=33, pair_coef=0.0, sigma=30.0, inertia=1.0, noise=0),
    dict(L=64, T=8, pair_coef=0.2, sigma=1.0, inertia=0.5, noise=2),
]


@pytest.mark.parametrize("mi", range(len(MODELS)))
def test_certified_labels_are_the_fp64_labels(mi):
    mod = MODELS[mi]
    L, T = mod["L"], mod["T"]
    rng = np.random.default_rng(100 + mi)
    n = 400
    mid = rng.integers(0, L, (n, 1))
    x = np.where(rng.random((n, 1)) < 0.4, rng.integers(0, L, (n, 4)),
                 np.clip(mid + rng.integers(-T - 2, T + 3, (n, 4)), 0, L - 1))
    x = np.where(rng.random((n, 4)) < 0.9, x, MISSING)    # missing: image border
    x[:4] = MISSING                                       # a single-pixel image
    g = np.where(rng.random(n) < 0.7, np.clip(mid[:, 0] + rng.integers(-20, 21, n), 0, L - 1),
                 rng.integers(0, L, n))
    xi = np.where(rng.random(n) < 0.7, np.clip(g + rng.integers(-9, 10, n), 0, L - 1),
                  rng.integers(0, L, n))
    g[4:8], xi[4:8] = [0, L - 1, 0, L - 1], [0, 0, L - 1, L - 1]
    C = _exact_cdf(mod, x, g, xi)
    Zx = C[:, -1]
    total = uncertain = 0
    for ulp in (-1.0, 0.0, 1.0):
        with np.errstate(invalid="ignore"):
            r = _prepare(mod, x, g, xi, ulp)
        # uniforms on and around every boundary the FP64 CDF has, and at random
        for k in list(range(0, L, max(1, L // 24))) + [-1]:
            b = np.floor(C[:, k] / Zx * 2.0 ** 24) if k >= 0 else rng.integers(0, 1 << 24, n)
            for o in (-2, -1, 0, 1, 2, 40, -40) if k >= 0 else (0,):
                ub = np.clip(b + o, 0, (1 << 24) - 1).astype(np.int64)
                s, certain, M = _draw(mod, r, g, xi, ub)
                want = (C <= (ub * 2.0 ** -24 * Zx)[:, None]).sum(1).clip(0, L - 1)
                assert (s[certain] == want[certain]).all()
                if k < 0:
                    total += n
                    uncertain += int((~certain).sum())
        # CDF values at the ends of the segments, within the margin (without
        # the share of the probed label and of t)
        at = np.arange(n)
        for i, (_, end) in enumerate(r["ends"][:-1]):
            lab = (end & 511) - 256 + g                    # last label of the segment
            ok = lab >= 0
            ref = np.where(ok, C[at, np.maximum(lab, 0)], 0.0) / Zx
            fin = np.isfinite(r["Z"])      # others certify nothing
            err = np.abs(r["Gd"][i].astype(f64) / r["Z"] - ref)
            bound = 1.25 * U * (r["E1"] + 0.6931472 * (r["E2"] - r["cb"] * r["Z"]) +
                                22 * r["Z"] + (1.39 * r["av"] + r["kd"]) * r["delta"]) / r["Z"]
            assert (err <= bound)[fin].all() and fin.mean() > 0.9
    assert uncertain < 0.05 * total


def test_a_dropped_term_is_caught():
    """The replay with the atom's join left out disagrees with the FP64 draw."""
    mod = MODELS[0]
    rng = np.random.default_rng(5)
    n, L = 400, mod["L"]
    mid = rng.integers(60, 200, (n, 1))
    x = mid + rng.integers(-20, 21, (n, 4))
    g = mid[:, 0] + rng.integers(-10, 11, n)
    xi = g.copy()
    C = _exact_cdf(mod, x, g, xi)
    r = _prepare(mod, x, g, xi, 0.0)
    r["delta"] = np.zeros(n, f32)
    ub = rng.integers(0, 1 << 24, n)
    s, certain, _ = _draw(mod, r, g, xi, ub)
    want = (C <= (ub * 2.0 ** -24 * C[:, -1])[:, None]).sum(1)
    assert (s[certain] != want[certain]).any()
