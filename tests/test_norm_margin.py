"""The Lp-price draw's per-site margin (csrc/pcad_device.cuh, draw_fp32_norm):
the FP32 draw replayed on the CPU with ex2 pushed 2 ulp either way.  Every draw
it calls certain picks the label of the oracle's FP64 inverse-CDF draw, for
uniforms on and around every boundary, and random draws are almost all
certain."""
import numpy as np
import pytest

f32, f64 = np.float32, np.float64
U = 2.0 ** -24


@pytest.fixture(scope="module")
def pc():
    import paper_2507_14869_gb300 as pc
    pc.lib()
    return pc


def fma(a, b, c):   # exact in FP64 for these factors, one rounding
    return (np.asarray(a, f64) * np.asarray(b, f64) + np.asarray(c, f64)).astype(f32)


def replay(mg, m, kappa, g, xi, nbrs, ub, ulp):
    L, p = m["L"], m["inertia_norm"]
    s = np.arange(L)
    P = sum(np.minimum(np.abs(s - x), m["T"]) for x in nbrs)
    c = f32(f64(-kappa) * abs(g - xi) ** p)
    t1 = fma(kappa, np.abs(s - xi) ** p, c)
    v = fma(f32(mg["alpha"]), (g - s) ** 2, fma(f32(mg["gam"]), P, t1))
    w = np.exp2(v.astype(f64)).astype(f32)
    w = (w.astype(f64) * (1.0 + np.where(s % 2 == 0, ulp, -ulp) * 2 * U)).astype(f32)
    G, comp, Gs, pre = f32(0), f32(0), [], []
    for b in range(0, L, 8):
        S, pp = f32(0), []
        for k in w[b:b + 8]:
            S = f32(S + k)
            pp.append(S)
        y = f32(S - comp)
        tt = f32(G + y)
        comp = f32(f32(tt - G) - y)
        G = tt
        Gs.append(G)
        pre.append(pp)
    lg = f32(np.log2(f64(G)))
    inner = fma(f32(2.3333335), c, f32(f32(1.3333334) * f32(f32(mg["hb"]) - lg)))
    eta = fma(f32(mg["kb1"]), inner, f32(mg["kb0"]))
    margin = f32(eta * G)
    labels, certain = [], []
    for u in ub:
        t = f32(f32(f32(u) * f32(U)) * G)
        cs = min(sum(int(x <= t) for x in Gs), len(Gs) - 1)
        Gp = Gs[cs - 1] if cs else f32(0)
        C = [f32(Gp + x) for x in pre[cs]]
        k = sum(int(x <= t) for x in C)
        found = k < len(C)
        k = min(k, len(C) - 1)
        lab = 8 * cs + k
        hi, lo = C[k], C[k - 1] if k else Gp
        labels.append(lab)
        certain.append(found and (lab == L - 1 or f32(hi - t) > margin)
                       and (lab == 0 or f32(t - lo) > margin))
    return np.array(labels), np.array(certain)


MODELS = [
    dict(L=33, nbhd=8, pair=0, pair_coef=0.833, pair_T=1, noise=0, sigma=3.2, inertia=2.0, inertia_norm=1),
    dict(L=16, nbhd=4, pair=1, pair_coef=0.4, pair_T=3, noise=0, sigma=1.5, inertia=12.0, inertia_norm=2),
    dict(L=100, nbhd=4, pair=1, pair_coef=0.1, pair_T=20, noise=0, sigma=9.0, inertia=30.0, inertia_norm=1),
    dict(L=5, nbhd=8, pair=0, pair_coef=0.2, pair_T=1, noise=0, sigma=0.8, inertia=0.1, inertia_norm=2),
]


@pytest.mark.parametrize("ulp", [-1.0, 0.0, 1.0])
@pytest.mark.parametrize("i", range(len(MODELS)))
def test_certain_draws_pick_the_fp64_label(pc, orc, i, ulp):
    m = dict(MODELS[i])
    m["T"] = 1 if m["pair"] == 0 else m["pair_T"]
    om = dict(m, flip_p=0.1, sampler=0)
    mg = pc.pcad_model_margins(om)
    L, lam = m["L"], m["inertia"]
    kappa = f32(-lam * 1.4426950408889634 / float(L - 1) ** m["inertia_norm"])
    rng = np.random.default_rng(900 + i)
    n_certain = 0
    for _ in range(40):
        g, xi = int(rng.integers(0, L)), int(rng.integers(0, L))
        nbrs = [int(v) for v in np.clip(xi + rng.integers(-4, 5, int(rng.integers(1, m["nbhd"] + 1))), 0, L - 1)]
        cdf = np.cumsum(orc.site_probs(om, g, xi, nbrs, lam))
        ub = list(rng.integers(0, 1 << 24, 32))
        for c in cdf[:-1]:
            ub += [min(max(int(c * (1 << 24)) + d, 0), (1 << 24) - 1)
                   for d in (-3, -1, 0, 1, 2, 20, -20, 60, -60, 400, -400)]
        labels, certain = replay(mg, m, kappa, g, xi, nbrs, ub, ulp)
        for u, lab, ok in zip(ub, labels, certain):
            if ok:
                want, _ = orc.site_draw(om, g, xi, nbrs, lam, u / float(1 << 24))
                assert lab == want, (g, xi, nbrs, u)
        n_certain += int(certain[:32].sum())
    assert n_certain > 0.99 * 32 * 40
