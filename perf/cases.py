"""What a user of the sampler has it do, as calls that can be timed.

A case is one pass through the public entry points: whole chains (reset, run,
read the sample and the posterior mean, PSNR / SSIM where a clean image is at
hand), the annealed restoration protocol, an uneven batch, and a server with a
backlog of requests.  Sizes, label counts and coefficients are those of the
repository's workloads (pcad_inputs, bench.py, protocol.py); the images are
seeded synthetic scenes of the same kind, made on the GPU.

``exact`` recomputes a case in 64 bits with plain torch: the keyed Philox
uniforms, the FP64 conditional of every label, the inverse CDF in label order.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_14869_gb300 as pc
from paper_2507_14869_gb300 import protocol

POTTS, TL = 0, 1
GAUSS, FLIP = 0, 1
PCA, GIBBS = 0, 1


def _chain(name, H, W, L, sweeps, burn_in, **kw):
    c = dict(name=name, path="chain", H=H, W=W, L=L, nbhd=4, sampler=PCA, sweeps=sweeps,
             burn_in=burn_in, pair=TL, pair_coef=0.05, pair_T=30, noise=GAUSS, sigma=20.0,
             flip_p=0.1, inertia=2.0, norm=0, track=False, score=False)
    c.update(kw)
    return c


_ISING = dict(pair=POTTS, pair_coef=1.2, pair_T=1, noise=FLIP, sigma=1.0, inertia=1.0)


def listed():
    return [
        # the binary 64 x 64 workload: the smallest call, one image of text or mask size
        _chain("binary64", 64, 64, 2, 500, 100, score=True, **_ISING),
        # its Gibbs comparison run
        _chain("binary64_gibbs", 64, 64, 2, 500, 100, sampler=GIBBS, **_ISING),
        # one annealed restoration of the paper's protocol, create to last sample
        dict(name="restore_l9", path="restore", side=256, L=9, sigma=0.2, q=0.46, sampler=PCA,
             stage_sweeps=250),
        # the same protocol by checkerboard Gibbs (four colour classes)
        dict(name="restore_l5_gibbs", path="restore", side=256, L=5, sigma=0.25, q=0.46,
             sampler=GIBBS, stage_sweeps=250),
        # the greyscale workload: a photograph-like 8-bit image, scored
        _chain("grey512", 512, 512, 256, 2000, 500, score=True),
        # its Gibbs comparison run
        _chain("grey512_gibbs", 512, 512, 256, 2000, 500, sampler=GIBBS),
        # the large image at few labels (a scan quantised to 16 levels), scored
        _chain("large_l16", 8192, 8192, 16, 200, 50, sigma=1.0, score=True),
        # the large image at all 8-bit labels: the benchmark's headline model
        _chain("large_l256", 8192, 8192, 256, 100, 25, sigma=25.0),
        # a large two-label mask of ragged width
        _chain("mask_2043x3001", 2043, 3001, 2, 200, 50, **_ISING),
        # MAP search: the price proportional to the change, every sweep's energy tracked
        _chain("map_search_l1", 301, 453, 33, 200, 50, nbhd=8, pair=POTTS, pair_coef=0.833,
               pair_T=1, sigma=3.2, inertia=2.0, norm=1, track=True),
        # uneven images of a set, two chains each, in one batch
        dict(name="batch_uneven", path="batch", mix=4, images=16, chains=2, lo=64, hi=1024,
             sweeps=200, burn_in=50),
        # a backlog of requests of different sizes and budgets on the server
        dict(name="serve_backlog", path="serve", mix=50, requests=10, lo=128, hi=1024,
             sweeps_lo=300, sweeps_hi=900),
    ]


# ---------------------------------------------------------------- models

def _image_params(rng, L):
    """Prior, noise and inertia of one image (the seeded table of the batch workload)."""
    s255 = rng.uniform(5.0, 40.0)
    if L == 2:
        return dict(pair=POTTS, pair_coef=2.0 * rng.uniform(0.4, 0.8), pair_T=1, noise=FLIP,
                    sigma=1.0, flip_p=s255 / 200.0, inertia=rng.uniform(0.5, 1.5))
    scale = 255.0 / (L - 1)
    return dict(pair=TL, pair_coef=rng.uniform(0.03, 0.08) * scale,
                pair_T=max(1, int(round(30.0 / scale))), noise=GAUSS, sigma=s255 / scale,
                flip_p=0.1, inertia=rng.uniform(1.0, 3.0))


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["chain"] * 6 + ["restore"] * 2 + ["batch", "serve"])
    if path == "restore":
        L = rng.choice([5, 9, 33])
        return dict(path="restore", side=_log(rng, 64, 512), L=L,
                    sigma={5: 0.25, 9: 0.2, 33: 0.1}[L], q=round(rng.uniform(0.06, 0.71), 2),
                    sampler=rng.choice([PCA, PCA, GIBBS]), stage_sweeps=rng.choice([100, 250]))
    if path == "batch":
        return dict(path="batch", mix=rng.randrange(1, 10 ** 6), images=rng.randrange(4, 17),
                    chains=rng.choice([1, 2, 4]), lo=64, hi=768,
                    sweeps=16 * rng.randrange(4, 13), burn_in=50)
    if path == "serve":
        return dict(path="serve", mix=rng.randrange(1, 10 ** 6), requests=rng.randrange(4, 11),
                    lo=128, hi=1024, sweeps_lo=300, sweeps_hi=600)
    # chains: sides from an icon to a scan, aspect 1 to 3, any label count
    H = _log(rng, 32, 4096)
    W = min(4096, int(round(H * rng.uniform(1.0, 3.0))))
    if rng.random() < 0.5:
        H, W = W, H
    kind = rng.choice(["two", "few", "few", "many", "grey", "grey"])
    L = {"two": 2, "few": rng.randrange(3, 17), "many": rng.randrange(17, 200), "grey": 256}[kind]
    c = _chain("", H, W, L, 100, 25, **_image_params(rng, L))
    del c["name"]
    c["nbhd"] = rng.choice([4, 4, 8])
    # the entry points take a prior range |pair_coef| nbhd T of at most 40
    c["pair_coef"] = min(c["pair_coef"], 38.0 / (c["nbhd"] * c["pair_T"]))
    c["sampler"] = rng.choice([PCA, PCA, GIBBS])
    c["score"] = rng.random() < 0.3
    most = min(1000, int(1.2e9 / (H * W)) if L > 16 else int(4e9 / (H * W)))
    c["sweeps"] = _log(rng, 50, max(51, most))
    c["burn_in"] = c["sweeps"] // 4
    return c


def _members(case):
    """The images of a batch or the requests of a server: sizes and models from the mix."""
    import random
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["images"] if case["path"] == "batch" else case["requests"]):
        H = _log(rng, case["lo"], case["hi"])
        if case["path"] == "batch":
            W = int(round(H * rng.uniform(1.0, 3.0)))
            if rng.random() < 0.5:
                H, W = W, H
            L = rng.choice([2, 16, 256])
            n, burn, chains = case["sweeps"], case["burn_in"], case["chains"]
        else:
            W, L = H, rng.choice([16, 256])
            n = rng.randrange(case["sweeps_lo"], case["sweeps_hi"] + 1)
            burn, chains = n // 4, 1
        for k in range(chains):
            p = _image_params(rng, L) if k == 0 else p
            out.append(dict(_chain("", H, W, L, n, burn, **p), image=len(out) - k, chain=k))
    return out


def _model(c):
    return dict(L=c["L"], nbhd=c["nbhd"], pair=c["pair"], pair_coef=c["pair_coef"],
                pair_T=c["pair_T"], noise=c["noise"], sigma=c["sigma"], flip_p=c["flip_p"],
                inertia=c["inertia"], sampler=c["sampler"], inertia_norm=c["norm"])


# ---------------------------------------------------------------- inputs

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _scene(seed, H, W, L):
    """Piecewise-constant shapes over a smooth gradient (two labels: over 0)."""
    rng = np.random.default_rng(seed)
    dev = _dev()
    top = float(L - 1)
    r = torch.arange(H, device=dev, dtype=torch.float32)[:, None]
    c = torch.arange(W, device=dev, dtype=torch.float32)[None, :]
    if L == 2:
        img = torch.zeros((H, W), device=dev)
    else:
        lo, hi = sorted(rng.uniform(0.0, top, 2))
        th, ph = rng.uniform(0.0, 2.0 * math.pi, 2)
        fr, fc = rng.uniform(0.5, 2.0, 2)
        ramp = math.cos(th) * r / max(H - 1, 1) + math.sin(th) * c / max(W - 1, 1)
        ramp = (ramp - ramp.min()) / max(float(ramp.max() - ramp.min()), 1e-12)
        img = lo + (hi - lo) * ramp + rng.uniform(0.05, 0.15) * top * torch.sin(
            2.0 * math.pi * (fr * r / max(H - 1, 1) + fc * c / max(W - 1, 1)) + ph)
    side = min(H, W)
    for _ in range(max(8, H * W // 16384) if L == 2 and H * W < 10 ** 6 else 20):
        y, x = int(rng.integers(0, H)), int(rng.integers(0, W))
        a, b = rng.integers(max(side // 16, 1), max(side // 4, 1) + 1, 2)
        v = float(rng.integers(0, 2)) if L == 2 else float(rng.uniform(0.0, top))
        y0, y1, x0, x1 = max(y - a, 0), min(y + a + 1, H), max(x - b, 0), min(x + b + 1, W)
        if rng.integers(0, 2):
            img[y0:y1, x0:x1] = v
        else:
            d = ((r[y0:y1] - y) / float(a)) ** 2 + ((c[:, x0:x1] - x) / float(b)) ** 2
            img[y0:y1, x0:x1] = torch.where(d <= 1.0, torch.full_like(d, v), img[y0:y1, x0:x1])
    return img.clamp_(0.0, top).round_()


def _image(case, seed):
    """(clean, noisy) label images in host memory, as a user's file gives them."""
    H, W, L = case["H"], case["W"], case["L"]
    img = _scene(seed, H, W, L)
    gen = torch.Generator(device=img.device)
    gen.manual_seed(seed + 7)
    if case["noise"] == FLIP:
        flips = torch.rand((H, W), device=img.device, generator=gen) < case["flip_p"]
        noisy = torch.where(flips, 1.0 - img, img)
    else:
        noise = torch.randn((H, W), device=img.device, generator=gen)
        noisy = (img + case["sigma"] * noise).clamp_(0.0, float(L - 1)).round_()
    return img.to(torch.uint8).cpu().numpy(), noisy.to(torch.uint8).cpu().numpy()


def _restore_image(case, seed):
    L = case["L"]
    return _image(dict(H=case["side"], W=case["side"], L=L, noise=GAUSS,
                       sigma=case["sigma"] * (L - 1)), seed)


def prepare(case, seed):
    s = dict(case=case)
    if case["path"] == "restore":
        s["g"] = _restore_image(case, seed)[1]
        s["seed"] = seed
        return s
    if case["path"] == "chain":
        clean, g = _image(case, seed)
        s["chain"] = pc.Chain(g, _model(case), seed=seed, chain_id=0, burn_in=case["burn_in"])
        if case["track"]:
            s["chain"].track_energy(case["sweeps"])
        s["clean"] = clean
        mean = torch.empty((case["H"], case["W"]), dtype=torch.float32,
                           pin_memory=torch.cuda.is_available())
        s["mean"] = mean.numpy()   # the caller's own pinned read-back buffer
        return s
    members = _members(case)
    images = {}
    for m in members:
        if m["image"] not in images:
            images[m["image"]] = _image(m, seed * 1000 + m["image"])[1]
    s["jobs"] = [(images[m["image"]], _model(m), seed + m["image"], m["chain"], m["burn_in"])
                 for m in members]
    if case["path"] == "batch":
        s["batch"] = _Batch(pc.pcad_batch_create(s["jobs"]))
    else:
        s["budgets"] = [m["sweeps"] for m in members]
        s["server"] = _Server(pc.pcad_server_create(256, 150 * 10 ** 9))
        pc.pcad_server_set_policy(s["server"].h, pc.SERVE_SRPT, 0.2)
    return s


class _Batch:
    """Frees the batch with the state that holds it."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        pc.pcad_batch_destroy(self.h)


class _Server:
    """Frees the server with the state that holds it."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        pc.pcad_server_destroy(self.h)


# ---------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    if case["path"] == "restore":
        return dict(sample=protocol.restore(
            state["g"], case["L"], J=1.0 / 3.0, q=case["q"], sigma=case["sigma"],
            seed=state["seed"], sampler=case["sampler"], stage_sweeps=case["stage_sweeps"]))
    if case["path"] == "chain":
        ch = state["chain"]
        ch.reset()
        ch.run(case["sweeps"])
        out = dict(sample=ch.sample(),
                   mean=pc.pcad_chain_read_mean(ch.h, case["H"], case["W"], out=state["mean"]))
        if case["score"]:
            out["psnr"], out["ssim"] = ch.metrics(state["clean"])
        if case["track"]:
            out["energies"] = ch.energies()
            out["best"], out["best_energy"], out["best_sweep"] = ch.min_state()
        return out
    jobs = state["jobs"]
    if case["path"] == "batch":
        b = state["batch"].h
        pc.pcad_batch_reset(b)
        pc.pcad_batch_run(b, case["sweeps"])
        pc.pcad_batch_sync(b)
        return [[pc.pcad_batch_read_sample(b, i, *g.shape) for i, (g, *_) in enumerate(jobs)],
                [pc.pcad_batch_read_mean(b, i, *g.shape) for i, (g, *_) in enumerate(jobs)]]
    sv = state["server"].h
    waiting = {}
    for i, (g, m, seed, chain, burn) in enumerate(jobs):
        waiting[pc.pcad_server_submit(sv, g, m, seed, chain, burn, state["budgets"][i])] = i
    out = [None] * len(jobs)
    while waiting:
        _, _, finished = pc.pcad_server_step(sv, 16)
        if not finished:
            continue
        for rid in list(waiting):
            i = waiting[rid]
            st, sample, mean = pc.pcad_server_poll(sv, rid, *jobs[i][0].shape)
            if st == 2:
                out[i] = [sample, mean]
                del waiting[rid]
    return out


# ---------------------------------------------------------------- floors and 64 bits

def _chains(case):
    """The chains of a case as chain cases."""
    if case["path"] == "chain":
        return [case]
    if case["path"] == "restore":
        return [dict(H=case["side"], W=case["side"], L=case["L"],
                     sweeps=4 * case["stage_sweeps"])]
    return _members(case)


def work(case):
    """An observation in, a sample out (and a mean, but for the restoration): the state can
    stay on the chip in between.  A draw needs a weight and a running sum per label."""
    out = 2 if case["path"] == "restore" else 6
    sites = [(c["H"] * c["W"], c["L"], c["sweeps"]) for c in _chains(case)]
    return dict(bytes=out * sum(n for n, _, _ in sites),
                flops=sum(2 * L * n * t for n, L, t in sites))


def _philox(H, W, row_words, sweep, chain, tag, seed, dev):
    """24-bit uniforms of the H x W sites: Philox4x32-10 keyed by (seed), counter (column
    group, row, sweep, tag and chain)."""
    m32 = 0xFFFFFFFF
    c0 = torch.arange(row_words, device=dev, dtype=torch.int64)[None, :].expand(H, row_words)
    c1 = torch.arange(H, device=dev, dtype=torch.int64)[:, None].expand(H, row_words)
    c2 = torch.full_like(c0, sweep)
    c3 = torch.full_like(c0, (tag << 24) | chain)
    k0, k1 = seed & m32, (seed >> 32) & m32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & m32) ^ c1 ^ k0, p1 & m32,
                          ((p0 >> 32) & m32) ^ c3 ^ k1, p0 & m32)
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return (torch.stack((c0, c1, c2, c3), -1).reshape(H, 4 * row_words)[:, :W] >> 8)


class _Exact:
    """One chain in FP64."""

    def __init__(self, g, m, seed, chain):
        self.dev = _dev()
        self.g = torch.from_numpy(g).to(self.dev).to(torch.int64)
        self.H, self.W = g.shape
        self.seed, self.chain, self.t = seed, chain, 0
        self.L = m["L"]
        # labels with a one-site border of the "missing" label L
        self.x = torch.full((self.H + 2, self.W + 2), self.L, device=self.dev, dtype=torch.int64)
        self.x[1:-1, 1:-1] = self.g
        self.offs = [(-1, 0), (1, 0), (0, -1), (0, 1)]
        if m["nbhd"] == 8:
            self.offs += [(-1, -1), (-1, 1), (1, -1), (1, 1)]
        self.set_model(m)

    def set_model(self, m):
        self.m, L, f = m, self.L, np.float32
        s = torch.arange(L, device=self.dev, dtype=torch.float64)
        d = (s[:, None] - s[None, :]).abs()
        T = 1.0 if m["pair"] == POTTS else float(m["pair_T"])
        V = float(f(m["pair_coef"])) * torch.clamp(d, max=T)   # Potts up to a constant
        self.E = torch.cat((torch.exp(-V), torch.ones((1, L), device=self.dev,
                                                      dtype=torch.float64)))
        if m["noise"] == FLIP:
            p = float(f(m["flip_p"]))
            self.U = torch.where(d == 0, -math.log(1.0 - p), -math.log(p)).to(torch.float64)
        else:
            self.U = d * d / (2.0 * float(f(m["sigma"])) ** 2)
        self.A = torch.exp(-self.U)
        lam = float(f(m["inertia"])) if m["sampler"] == PCA else 0.0
        n = m.get("inertia_norm", 0) if L > 2 else 0
        self.I = torch.exp(-lam * ((d > 0).to(torch.float64) if n == 0 else (d / (L - 1)) ** n))

    def _draw(self, r, c, u):
        """New labels of the sites at rows r, columns c (flat indices, u the uniforms)."""
        w = self.A[self.g[r, c]]
        for dr, dc in self.offs:
            w *= self.E[self.x[r + 1 + dr, c + 1 + dc]]
        if self.m["sampler"] == PCA:
            w *= self.I[self.x[r + 1, c + 1]]
        C = torch.cumsum(w, -1)
        t = u.to(torch.float64) * 2.0 ** -24 * C[:, -1]
        return (C <= t[:, None]).sum(-1).clamp_(max=self.L - 1)

    def sweep(self):
        H, W = self.H, self.W
        gibbs = self.m["sampler"] == GIBBS
        u = _philox(H, W, (W + 3) // 4, self.t, self.chain, int(gibbs), self.seed, self.dev)
        step = max(1, (1 << 26) // (W * self.L))
        if not gibbs:
            new = torch.empty_like(self.g)
            c0 = torch.arange(W, device=self.dev)
            for y in range(0, H, step):
                n = min(step, H - y)
                r = torch.arange(y, y + n, device=self.dev).repeat_interleave(W)
                new[y:y + n] = self._draw(r, c0.repeat(n), u[y:y + n].reshape(-1)).reshape(n, W)
            self.x[1:-1, 1:-1] = new
        else:
            if not hasattr(self, "colours"):
                rr = torch.arange(H, device=self.dev)[:, None]
                cc = torch.arange(W, device=self.dev)[None, :]
                col = (rr + cc) % 2 if self.m["nbhd"] == 4 else 2 * (rr % 2) + cc % 2
                self.colours = [torch.nonzero(col == q, as_tuple=True)
                                for q in range(2 if self.m["nbhd"] == 4 else 4)]
            for r, c in self.colours:
                for k in range(0, len(r), step * W):
                    a, b = r[k:k + step * W], c[k:k + step * W]
                    self.x[a + 1, b + 1] = self._draw(a, b, u[a, b])
        self.t += 1

    def labels(self):
        return self.x[1:-1, 1:-1]

    def energy(self):
        """Posterior energy: every neighbour pair once, the Potts reward per equal pair."""
        x, m = self.labels(), self.m
        c = float(np.float32(m["pair_coef"]))
        s = 0.0
        for dr, dc in [(0, 1), (1, 0)] + ([(1, 1), (1, -1)] if m["nbhd"] == 8 else []):
            a, b = x[:x.shape[0] - dr], x[dr:]
            a, b = (a[:, :a.shape[1] - 1], b[:, 1:]) if dc == 1 else \
                (a[:, 1:], b[:, :b.shape[1] - 1]) if dc == -1 else (a, b)
            d = (a - b).abs()
            s += -c * float((d == 0).sum()) if m["pair"] == POTTS else \
                c * float(d.clamp(max=m["pair_T"]).sum())
        return s + float(self.U[self.g, x].sum())


def _scores(mean, clean, L):
    """PSNR and mean SSIM (11 x 11 Gaussian window, sigma 1.5) of a posterior mean."""
    x = torch.from_numpy(clean).to(mean.device).to(torch.float64) / (L - 1)
    y = mean / (L - 1)
    mse = float(((x - y) ** 2).mean())
    psnr = math.inf if mse == 0.0 else 20.0 * math.log10(float(x.max()) / math.sqrt(mse))
    if min(x.shape) < 11:
        n = x.numel()
        mx, my = x.mean(), y.mean()
        vx, vy = ((x - mx) ** 2).sum() / (n - 1), ((y - my) ** 2).sum() / (n - 1)
        cxy = ((x - mx) * (y - my)).sum() / (n - 1)
        return psnr, float((2 * mx * my + 1e-4) * (2 * cxy + 9e-4) /
                           ((mx * mx + my * my + 1e-4) * (vx + vy + 9e-4)))
    w = [math.exp(-(a - 5.0) ** 2 / 4.5) for a in range(11)]
    w = [a / sum(w) for a in w]

    def blur(v):
        v = sum(w[a] * v[a:v.shape[0] - 10 + a] for a in range(11))
        return sum(w[a] * v[:, a:v.shape[1] - 10 + a] for a in range(11))
    total, n = 0.0, 0
    for r in range(0, x.shape[0] - 10, 1024):   # bands of rows keep it small
        a, b = x[r:r + 1034], y[r:r + 1034]
        mx, my = blur(a), blur(b)
        v = (2 * mx * my + 1e-4) * (2 * (blur(a * b) - mx * my) + 9e-4) / (
            (mx * mx + my * my + 1e-4) *
            (blur(a * a) - mx * mx + blur(b * b) - my * my + 9e-4))
        total, n = total + float(v.sum()), n + v.numel()
    return psnr, total / n


def _exact_chain(c, g, m, seed, chain, track=False):
    e = _Exact(g, m, seed, chain)
    acc = torch.zeros(g.shape, device=e.dev, dtype=torch.int64)
    energies, best = [], None
    for t in range(c["sweeps"]):
        e.sweep()
        if t >= c["burn_in"]:
            acc += e.labels()
        if track:
            energies.append(e.energy())
            if best is None or energies[-1] < best[1]:
                best = (e.labels().clone(), energies[-1], t + 1)
    mean = acc.to(torch.float64) / (c["sweeps"] - c["burn_in"])
    return e.labels().to(torch.uint8), mean, energies, best


def exact(case, seed):
    # about 20 seconds of 64-bit label evaluations and of small launches
    if sum(c["H"] * c["W"] * c["L"] * c["sweeps"] for c in _chains(case)) > 2.5e11 or \
            sum(c["sweeps"] for c in _chains(case)) > 8000:
        return None
    if case["path"] == "restore":
        L, J, q, n = case["L"], 1.0 / 3.0, case["q"], case["stage_sweeps"]
        ms = [dict(L=L, nbhd=8, pair=POTTS, pair_coef=2.0 * b * J, pair_T=1, noise=GAUSS,
                   sigma=case["sigma"] * (L - 1), flip_p=0.1, inertia=b * q,
                   sampler=case["sampler"]) for b in (1.25, 1.5, 1.75, 2.0)]
        e = _Exact(_restore_image(case, seed)[1], ms[0], seed, 0)
        for m in ms:
            e.set_model(m)
            for _ in range(n):
                e.sweep()
        return dict(sample=e.labels().to(torch.uint8))
    if case["path"] == "chain":
        clean, g = _image(case, seed)
        x, mean, energies, best = _exact_chain(case, g, _model(case), seed, 0, case["track"])
        out = dict(sample=x, mean=mean)
        if case["score"]:
            out["psnr"], out["ssim"] = _scores(mean, clean, case["L"])
        if case["track"]:
            out["energies"] = np.array(energies, dtype=np.float64)
            out["best"], out["best_energy"], out["best_sweep"] = best[0].to(torch.uint8), *best[1:]
        return out
    res, images = [], {}
    for m in _members(case):
        if m["image"] not in images:
            images[m["image"]] = _image(m, seed * 1000 + m["image"])[1]
        x, mean, _, _ = _exact_chain(m, images[m["image"]], _model(m), seed + m["image"],
                                     m["chain"])
        res.append([x, mean])
    return res if case["path"] == "serve" else [[r[0] for r in res], [r[1] for r in res]]
