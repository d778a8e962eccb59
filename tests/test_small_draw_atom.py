"""The small-label draw with the inertia atom joined to w(x_i) and to the chunk
prefixes (csrc/small_draw.cuh), replayed in FP32 on the CPU with ex2 pushed 2
ulp either way: every draw the replay calls certain picks the label of the
oracle's FP64 inverse-CDF draw, for uniforms on and around every boundary, and
random draws are almost all certain."""
import numpy as np
import pytest

f32, f64 = np.float32, np.float64
U = 2.0 ** -24


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


def replay(mg, model, g, xi, nbrs, ub, ulp, lmax):
    L, T = model["L"], model["T"]
    s = np.arange(lmax)
    P = np.zeros(lmax, np.int64)
    for x in nbrs:
        P += np.minimum(np.abs(s - x), T)
    aq = (f64(f32(mg["alpha"])) * (g - s) ** 2).astype(f32)
    v = (f64(f32(mg["gam"])) * P + aq.astype(f64)).astype(f32)
    w = np.exp2(v.astype(f64)).astype(f32)
    w = (w.astype(f64) * (1.0 + np.where(s % 2 == 0, ulp, -ulp) * 2 * U)).astype(f32)
    w[s >= L] = f32(0.0)
    S = [f32(f32(w[4 * c] + w[4 * c + 2]) + f32(w[4 * c + 1] + w[4 * c + 3]))
         for c in range(lmax // 4)]
    delta = f32(0.0)
    if model["inertia"] > 0:
        delta = f32(w[xi] * f32(np.expm1(f64(f32(model["inertia"])))))
        w[xi] = f32(w[xi] + delta)
    G = [S[0]]
    for c in range(1, lmax // 4):
        G.append(f32(G[-1] + S[c]))
    G = [f32(x + delta) if 4 * c + 3 >= xi else x for c, x in enumerate(G)]
    Z = G[-1]
    lg = f32(np.log2(f64(Z)))
    inner = f32(f64(f32(mg["kb1"])) * f64(f32(f32(mg["hb"]) - lg)) + f64(f32(mg["kb0"])))
    margin = f32(f64(inner) * f64(Z) + f64(f32(f32(mg["kbr"]) * delta)))
    labels, certain = [], []
    for u in ub:
        t = f32(f32(u) * f32(Z * f32(U)))
        cs = sum(int(x <= t) for x in G[:-1])
        Gp = G[cs - 1] if cs else f32(0.0)
        C = []
        for k in range(4):
            C.append(f32((C[-1] if k else Gp) + w[4 * cs + k]))
        k = sum(int(x <= t) for x in C[:3])
        hi, lo = C[k], C[k - 1] if k else Gp
        labels.append(4 * cs + k)
        certain.append(min(f32(hi - t), f32(t - lo)) > margin)
    return np.array(labels), np.array(certain)


MODELS = [
    dict(L=16, nbhd=4, pair=1, pair_coef=0.05, pair_T=30, noise=0, sigma=1.0, inertia=2.0),
    dict(L=16, nbhd=4, pair=1, pair_coef=1.36, pair_T=2, noise=0, sigma=2.3, inertia=3.0),
    dict(L=13, nbhd=8, pair=1, pair_coef=0.4, pair_T=3, noise=0, sigma=1.5, inertia=0.7),
    dict(L=16, nbhd=4, pair=1, pair_coef=0.3, pair_T=6, noise=0, sigma=3.0, inertia=0.0),
    dict(L=5, nbhd=8, pair=0, pair_coef=0.833, pair_T=1, noise=0, sigma=1.0, inertia=0.7),
    dict(L=3, nbhd=4, pair=1, pair_coef=0.5, pair_T=1, noise=0, sigma=0.7, inertia=20.0),
]


@pytest.mark.parametrize("ulp", [-1.0, 0.0, 1.0])
@pytest.mark.parametrize("i", range(len(MODELS)))
def test_certain_draws_pick_the_fp64_label(pc, orc, i, ulp):
    model = dict(MODELS[i])
    model["T"] = 1 if model["pair"] == 0 else model["pair_T"]
    om = dict(model, flip_p=0.1, sampler=0)
    mg = pc.pcad_model_margins(om)
    L, nbhd = model["L"], model["nbhd"]
    lmax = 8 if L <= 8 else 16
    rng = np.random.default_rng(700 + i)
    n_rand = n_certain = 0
    for _ in range(40):
        g, xi = int(rng.integers(0, L)), int(rng.integers(0, L))
        nn = int(rng.integers(1, nbhd + 1))
        nbrs = [int(v) for v in np.clip(xi + rng.integers(-3, 4, nn), 0, L - 1)]
        cdf = np.cumsum(orc.site_probs(om, g, xi, nbrs, model["inertia"]))
        ub = list(rng.integers(0, 1 << 24, 32))
        for c in cdf[:-1]:
            ub += [min(max(int(c * (1 << 24)) + d, 0), (1 << 24) - 1)
                   for d in (-3, -1, 0, 1, 2, 20, -20, 60, -60, 400, -400)]
        labels, certain = replay(mg, model, g, xi, nbrs, ub, ulp, lmax)
        for u, lab, ok in zip(ub, labels, certain):
            if ok:
                want, _ = orc.site_draw(om, g, xi, nbrs, model["inertia"], u / float(1 << 24))
                assert lab == want, (g, xi, nbrs, u)
        n_rand += 32
        n_certain += int(certain[:32].sum())
    assert n_certain > 0.99 * n_rand
