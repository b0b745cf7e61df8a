"""The work that a user of the library has it do, as measurable cases.

A survey program keeps one context and takes star after star through it: detrend the raw
light curve, fold and score it at every trial period of a grid, read off the decision;
many stars at once go through the batched search. Beside that stand the folds that return
profiles, the scorers on folded profiles, the generation of training profiles and a
training step of the CNN scorer. Light curves have Kepler's long cadence (29.4 minutes);
lengths, grids, bin counts and box widths are those of the tests, the benchmark and the
batched workload.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2312_02063_gb300 as g
from paper_2312_02063_gb300 import train as gtrain

CADENCE_D = 29.4 / 1440.0
CNN_FLOPS = 3_056_128.0  # multiply-adds x 2 of one profile's forward pass
SPACINGS = (0.5, 1.0, 1.5, 2.0, 3.0)


def listed():
    return [
        # a quick look at one quarter of data: the smallest search, bound by launches
        dict(name="search_tiny", kind="search", n_cad=4096, gaps=0.0, n_periods=2000, grid="freq", nbins=64,
             scorer="box", w_max=8),
        # one star over the whole mission at the densest grid, box detector
        dict(name="search_box_kepler", kind="search", n_cad=65536, gaps=0.04, n_periods=250000, grid="freq",
             nbins=256, scorer="box", w_max=108),
        # the paper's search: 100,000 periods uniform in period, CNN scorer
        dict(name="search_cnn_paper", kind="search", n_cad=65536, gaps=0.04, n_periods=100000, grid="period",
             nbins=256, scorer="cnn", w_max=0),
        # folded profiles for inspection: an odd length, an odd grid, bins not a power of two
        dict(name="fold_ragged", kind="fold", n_cad=30011, gaps=0.04, n_periods=12345, grid="freq", nbins=200),
        # the paper's own two-tier equal-count fold
        dict(name="equal_count_paper", kind="equal", n_cad=65536, gaps=0.04, n_periods=100000, grid="period",
             nfine=4096, nbins=256),
        # detection statistics: many short stars on a coarse grid, box detector
        dict(name="batch_short_box", kind="batch", stars=1024, n_lo=4096, n_hi=4096, p_lo=2000, p_hi=2000, nbins=256,
             scorer="box", w_max=160),
        # a survey batch: stars and grids of uneven length, CNN scorer
        dict(name="batch_uneven_cnn", kind="batch", stars=16, n_lo=8192, n_hi=70000, p_lo=20000, p_hi=250000,
             nbins=256, scorer="cnn", w_max=0),
        # stored profiles scored by each detector
        dict(name="score_box", kind="score_box", n=262144, nbins=256, w_max=32),
        dict(name="score_cnn", kind="score_cnn", n=262144),
        # one training step on a resident batch, and the batch's generation
        dict(name="train_step", kind="train", batch=4096),
        dict(name="synth_profiles", kind="synth", n=4096, n_cad=65536, nbins=256),
        # a raw full-length light curve made ready for the search
        dict(name="detrend_kepler", kind="detrend", n_cad=65536, gaps=0.04),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "fold", "equal", "batch", "score_box", "score_cnn", "train", "synth",
                       "detrend"])
    n_cad = _log(rng, 1000, 70000)
    gaps = rng.choice([0.0, 0.04])
    grid = rng.choice(["freq", "period"])
    if kind == "search":
        scorer = rng.choice(["box", "cnn"])
        nbins = 256 if scorer == "cnn" else rng.choice([64, 100, 128, 200, 256, 300, 512])
        return dict(kind=kind, n_cad=n_cad, gaps=gaps, n_periods=_log(rng, 500, 220000), grid=grid, nbins=nbins,
                    scorer=scorer, w_max=max(1, int(nbins * rng.uniform(0.1, 0.45))) if scorer == "box" else 0)
    if kind == "fold":
        return dict(kind=kind, n_cad=n_cad, gaps=gaps, n_periods=_log(rng, 500, 60000), grid=grid,
                    nbins=rng.choice([64, 100, 128, 200, 256, 300, 512, 1000]))
    if kind == "equal":
        return dict(kind=kind, n_cad=n_cad, gaps=gaps, n_periods=_log(rng, 500, 100000), grid=grid,
                    nfine=rng.choice([1000, 2048, 4096]), nbins=rng.choice([64, 100, 256]))
    if kind == "batch":
        scorer = rng.choice(["box", "cnn"])
        if rng.random() < 0.5:
            return dict(kind=kind, stars=_log(rng, 64, 1024), n_lo=1024, n_hi=_log(rng, 1500, 8192), p_lo=200,
                        p_hi=_log(rng, 300, 4000), nbins=256, scorer=scorer, w_max=160 if scorer == "box" else 0)
        return dict(kind=kind, stars=_log(rng, 2, 12), n_lo=8192, n_hi=70000, p_lo=20000, p_hi=250000, nbins=256,
                    scorer=scorer, w_max=108 if scorer == "box" else 0)
    if kind == "score_box":
        nbins = rng.choice([64, 100, 256, 300, 512])
        return dict(kind=kind, n=_log(rng, 300, 262144), nbins=nbins, w_max=max(1, int(nbins * rng.uniform(0.05, 0.45))))
    if kind == "score_cnn":
        return dict(kind=kind, n=_log(rng, 100, 262144))
    if kind == "train":
        return dict(kind=kind, batch=_log(rng, 100, 4096))
    if kind == "synth":
        return dict(kind=kind, n=_log(rng, 64, 4096), n_cad=n_cad, nbins=rng.choice([64, 200, 256]))
    return dict(kind=kind, n_cad=_log(rng, 4000, 70000), gaps=0.04)


# ---------------------------------------------------------------- inputs

_context = None


def _ctx():
    """The program's one context (and its workspace), kept from star to star."""
    global _context
    if _context is None:
        _context = g.Context(0)
    return _context


def _grid(n, form):
    if form == "period":
        return np.linspace(0.2, 1.0, n)
    k = np.arange(n, dtype=np.float64)
    return 1.0 / (1.0 + k * 4.0 / max(1, n - 1))


def _dips(t, period, epoch, duration):
    d = np.mod(t - epoch + 0.5 * period, period) - 0.5 * period
    return np.abs(d) < 0.5 * duration


def _light_curve(rng, shape, n_cad, gaps, sigma=2e-4, red=5e-5):
    """White and AR(1) noise, one injected transit; gaps of 1 to 5 days, which follow from `shape` and so
    belong to the case (the downtimes of the telescope), while the values follow from the seed."""
    t = np.arange(n_cad, dtype=np.float64) * CADENCE_D
    keep = np.ones(n_cad, bool)
    while (~keep).mean() < gaps:
        a = int(shape.uniform(0.0, n_cad))
        keep[a:a + int(shape.uniform(1.0, 5.0) / CADENCE_D) + 1] = False
    flux = 1.0 + rng.normal(0.0, sigma, n_cad)
    kernel = 0.9 ** np.arange(120)
    flux += np.convolve(rng.normal(0.0, red * math.sqrt(1 - 0.81), n_cad), kernel)[:n_cad]
    period = rng.uniform(0.2, 1.0)
    truth = (period, rng.uniform(0.0, period), rng.uniform(0.5, 2.0) / 24.0)
    depth = 1e-6 * math.exp(rng.uniform(math.log(50.0), math.log(500.0)))
    flux *= np.where(_dips(t, *truth), 1.0 - depth, 1.0)
    return t[keep], flux[keep].astype(np.float32), truth


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _profiles(seed, n, nbins):
    """Folded profiles and counts: half boxes, half noise or a sinusoid."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((n, 6), generator=gen, device="cuda")
    x = torch.arange(nbins, device="cuda")[None, :] / nbins
    sigma = 10.0 ** (-5.0 + 2.0 * u[:, :1])
    prof = torch.randn((n, nbins), generator=gen, device="cuda") * sigma
    depth = 3e-5 * (2000.0 / 30.0) ** u[:, 1:2]
    width = 0.02 + 0.3 * u[:, 2:3] ** 2
    box = ((x - u[:, 3:4]) % 1.0) < width
    kind = (u[:, 4:5] * 4).int()
    prof = prof - torch.where((kind < 2) & box, depth, torch.zeros_like(depth))
    wave = 1e-3 * 0.1 ** u[:, 1:2] * torch.sin(2 * math.pi * (x * (1 + 4 * u[:, 2:3]) + u[:, 3:4]))
    prof = (1.0 + prof + torch.where(kind == 3, wave, torch.zeros_like(wave))).float().contiguous()
    counts = (245 + 8 * torch.randn((n, nbins), generator=gen, device="cuda")).round().clamp_(1).int().contiguous()
    return prof, counts, (kind < 2).float().reshape(-1).contiguous()


def _weights(seed):
    w = gtrain.init_weights("cuda", seed)
    gen = torch.Generator(device="cuda").manual_seed(seed + 7)
    for n in w:
        if n.endswith(".b"):
            w[n].copy_(0.02 * torch.randn(w[n].shape, generator=gen, device="cuda"))
    return w


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    shape = np.random.Generator(np.random.PCG64(20235204))
    st = {"case": case, "ctx": _ctx()}
    if kind in ("search", "fold", "equal"):
        t, f, _ = _light_curve(rng, shape, case["n_cad"], case["gaps"])
        st.update(t=_dev(t), f=_dev(f), p=_dev(_grid(case["n_periods"], case["grid"])), t0=0.0)
    elif kind == "batch":
        ts, fs, ps = [], [], []
        for _ in range(case["stars"]):
            n = int(shape.integers(case["n_lo"], case["n_hi"] + 1))
            t, f, _ = _light_curve(rng, shape, n, 0.04, sigma=10.0 ** rng.uniform(-4.0, -3.0), red=0.0)
            ts.append(t)
            fs.append(f)
            ps.append(_grid(int(shape.integers(case["p_lo"], case["p_hi"] + 1)), "freq"))
        off = lambda xs: _dev(np.concatenate([[0], np.cumsum([len(x) for x in xs])]).astype(np.int64))  # noqa: E731
        st.update(lc=off(ts), go=off(ps), t=_dev(np.concatenate(ts)), f=_dev(np.concatenate(fs)),
                  p=_dev(np.concatenate(ps)), t0s=torch.zeros(case["stars"], dtype=torch.float64, device="cuda"),
                  lens=[len(x) for x in ts], grids=[len(x) for x in ps])
    elif kind in ("score_box", "score_cnn", "train"):
        n = case["batch"] if kind == "train" else case["n"]
        st["prof"], st["counts"], st["label"] = _profiles(int(seed), n, case.get("nbins", 256))
    elif kind == "synth":
        st["seed"] = int(seed)
        st["params"] = dict(g.TRAINING_SET, n_cadences=case["n_cad"])
    elif kind == "detrend":
        t, f, truth = _light_curve(rng, shape, case["n_cad"], case["gaps"])
        f = f.astype(np.float64) * (1.0 + 1e-3 * np.sin(2 * np.pi * t / rng.uniform(3.0, 8.0))
                                    + 4e-4 * np.sin(2 * np.pi * t / rng.uniform(0.8, 1.2)))
        f[rng.choice(len(t), 40, replace=False)] += 2e-3 * rng.choice([-1.0, 1.0], 40)
        st.update(t=_dev(t), f=_dev(f.astype(np.float32)), mask=_dev(_dips(t, truth[0], truth[1], 2 * truth[2]).astype(np.uint8)))
    if case.get("scorer") == "cnn" or kind in ("score_cnn", "train"):
        st["w"] = _weights(int(seed) % 1000003)
    if kind == "train":  # a run well under way: moments as after a hundred steps
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        st["m"] = {n: 1e-3 * torch.randn(t.shape, generator=gen, device="cuda") for n, t in st["w"].items()}
        st["v"] = {n: 1e-4 * (0.5 + torch.rand(t.shape, generator=gen, device="cuda")) for n, t in st["w"].items()}
        st["step"] = 100
    return st


# ---------------------------------------------------------------- the calls

def _decision(ctx, score, periods, offsets=None):
    """The decision on each star, as views of its records: FP64 statistics, the best peak, the number of peaks."""
    summary, _ = g.gpfc_peaks(ctx, score, periods, offsets, max_peaks=0)
    s = summary.numel() // g.STAR_SUMMARY_DTYPE.itemsize
    return {"sde_mean_sd": summary.view(torch.float64).view(s, 6)[:, :3],
            "best_index": summary.view(torch.int64).view(s, 6)[:, 3],
            "best_score": summary.view(torch.float32).view(s, 12)[:, 8],
            "n_peaks": summary.view(torch.int32).view(s, 12)[:, 9]}


def run(state):
    c, ctx = state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "search":
        kw = dict(scorer=g.SCORER_BOX, w_max=c["w_max"]) if c["scorer"] == "box" else \
            dict(scorer=g.SCORER_CNN, weights=state["w"])
        score, bi, bs = g.gpfc_search(ctx, state["t"], state["f"], state["p"], c["nbins"], state["t0"], **kw)
        return {"score": score, "best_index": bi, "best_score": bs, "star": _decision(ctx, score, state["p"])}
    if kind == "batch":
        kw = dict(scorer=g.SCORER_BOX, w_max=c["w_max"]) if c["scorer"] == "box" else \
            dict(scorer=g.SCORER_CNN, weights=state["w"])
        score, bi, bs = g.gpfc_search_batched(ctx, state["lc"], state["t"], state["f"], state["go"], state["p"],
                                              c["nbins"], state["t0s"], **kw)
        return {"score": score, "best_index": bi, "best_score": bs,
                "star": _decision(ctx, score, state["p"], state["go"])}
    if kind == "fold":
        folded, counts = g.gpfc_fold(ctx, state["t"], state["f"], state["p"], c["nbins"], state["t0"])
        return {"folded": folded, "counts": counts}
    if kind == "equal":
        return {"folded": g.gpfc_fold_equal_count(ctx, state["t"], state["f"], state["p"], c["nbins"], c["nfine"],
                                                  state["t0"])}
    if kind == "score_box":
        score, bs, bw = g.gpfc_score_box(ctx, state["prof"], state["counts"], 1, c["w_max"], 1.0)
        return {"score": score, "best_s": bs, "best_w": bw}
    if kind == "score_cnn":
        return {"score": g.gpfc_score_cnn(ctx, state["prof"], state["w"], state["counts"])}
    if kind == "train":
        w = state["w"]
        logit, saved = g.gpfc_cnn_forward_train(ctx, state["prof"], w, state["counts"])
        loss, dl = g.gpfc_bce_with_logits(ctx, logit, state["label"])
        grads = g.gpfc_cnn_backward(ctx, dl, w, saved)
        state["step"] += 1
        for n in g.CNN_PARAM_NAMES:
            g.gpfc_adam(ctx, w[n], grads[n], state["m"][n], state["v"][n], state["step"], 1e-3)
        return {"logit": logit, "loss": loss, "grads": grads, "weights": w}
    if kind == "synth":
        f, cn, y, per, sd = g.gpfc_synth_profiles(ctx, state["seed"], 0, c["n"], c["nbins"], state["params"],
                                                  want_period=True, want_std=True)
        return {"folded": f, "counts": cn, "label": y, "period": per, "flux_std": sd}
    t, f, s = g.gpfc_detrend(ctx, state["t"], state["f"], state["mask"])
    return {"times": t, "flux": f, "segment": s}


def work(case):
    """Inputs read once, outputs written once; two additions and three multiply-adds per sample and period
    (phase and accumulation), eight operations per box, the CNN's multiply-adds."""
    c, kind = case, case["kind"]

    def score_flops(np_, nbins, scorer, w_max):
        return np_ * (CNN_FLOPS if scorer == "cnn" else 8.0 * nbins * w_max)

    if kind in ("search", "fold", "equal"):
        n, P = c["n_cad"] * (1 - c["gaps"]), c["n_periods"]
        b, fl = n * 12 + P * 8, 8.0 * n * P
        if kind == "search":
            return {"bytes": b + 4 * P, "flops": fl + score_flops(P, c["nbins"], c["scorer"], c["w_max"])}
        return {"bytes": b + P * c["nbins"] * (8 if kind == "fold" else 4), "flops": fl}
    if kind == "batch":
        n, P = 0.96 * (c["n_lo"] + c["n_hi"]) / 2, (c["p_lo"] + c["p_hi"]) / 2
        return {"bytes": c["stars"] * (n * 12 + P * 12),
                "flops": c["stars"] * (8.0 * n * P + score_flops(P, c["nbins"], c["scorer"], c["w_max"]))}
    if kind == "score_box":
        return {"bytes": c["n"] * (8.0 * c["nbins"] + 12), "flops": score_flops(c["n"], c["nbins"], "box", c["w_max"])}
    if kind == "score_cnn":
        return {"bytes": c["n"] * (8.0 * 256 + 4), "flops": CNN_FLOPS * c["n"]}
    if kind == "train":
        return {"bytes": c["batch"] * (8.0 * 256 + 8) + 28.0 * 538_000, "flops": 3 * CNN_FLOPS * c["batch"]}
    if kind == "synth":  # per sample: a quarter of ten Philox rounds, Box-Muller, phase, accumulation
        return {"bytes": c["n"] * (8.0 * c["nbins"] + 16), "flops": 40.0 * c["n"] * c["n_cad"]}
    n = c["n_cad"] * (1 - c["gaps"])  # five spacings, a few fits each, some 40 operations a point and fit
    return {"bytes": n * 29.0, "flops": 5 * 4 * 40.0 * n}


# ---------------------------------------------------------------- 64-bit values

def _quantised(t, f, t0):
    """tau (units of 2^-24 d from the phase origin) and the flux about its mean, with the mean."""
    tau = torch.round((t - t0) * 16777216.0).to(torch.int64)
    f = f.double()
    ref = f.mean()
    return tau, f - ref, ref


def _bins(tau, p, nbins):
    """Bins of every sample at every period of p, [len(p)][n]: the 64-bit fixed-point phase times nbins."""
    F = torch.round(1099511627776.0 / p).to(torch.int64)
    phase = F[:, None] * tau[None, :]
    hi, lo = (phase >> 32) & 0xFFFFFFFF, phase & 0xFFFFFFFF
    return (hi * nbins + ((lo * nbins) >> 32)) >> 32


def _folds(tau, x, p, nbins, each=1 << 26):
    """(first period, sums, counts) of successive chunks of periods, in 64 bits."""
    step = max(1, each // max(len(tau), nbins))
    for a in range(0, len(p), step):
        b = _bins(tau, p[a:a + step], nbins)
        k = b.shape[0]
        b += nbins * torch.arange(k, device=b.device)[:, None]
        b = b.reshape(-1)
        s = torch.zeros(k * nbins, dtype=torch.float64, device=b.device)
        c = torch.zeros(k * nbins, dtype=torch.float64, device=b.device)
        s.scatter_add_(0, b, x.repeat(k))
        c.scatter_add_(0, b, torch.ones(1, dtype=torch.float64, device=b.device).expand(b.numel()))
        yield a, s.view(k, nbins), c.view(k, nbins)


def _box(s, c, w_max, sigma):
    """Largest box SNR of each profile."""
    S, N = s.sum(1, keepdim=True), c.sum(1, keepdim=True)
    zero = torch.zeros_like(S)
    ps = torch.cat([zero, torch.cat([s, s[:, :w_max]], 1).cumsum(1)], 1)
    pc = torch.cat([zero, torch.cat([c, c[:, :w_max]], 1).cumsum(1)], 1)
    n = s.shape[1]
    best = torch.full((s.shape[0],), -math.inf, dtype=torch.float64, device=s.device)
    for w in range(1, w_max + 1):
        si, ni = ps[:, w:w + n] - ps[:, :n], pc[:, w:w + n] - pc[:, :n]
        no = N - ni
        v = (S * ni - si * N) / torch.sqrt(N * ni * no)
        v = torch.where((ni >= 1) & (no >= 1), v, torch.full_like(v, -math.inf))
        best = torch.maximum(best, v.max(1).values)
    return best / sigma


def _conv(x, w, b):
    """Circular convolution with five taps, padding 2."""
    cols = torch.cat([torch.roll(x, 2 - j, 2) for j in range(5)], 1)
    return torch.matmul(w.permute(0, 2, 1).reshape(w.shape[0], -1), cols) + b[None, :, None]


def _logits(m, c, w):
    """The CNN in 64 bits on profiles m (means) with counts c."""
    full = c > 0
    n = full.sum(1, keepdim=True).clamp(min=1)
    v = torch.where(full, m, torch.zeros_like(m))
    mean = v.sum(1, keepdim=True) / n
    sd = torch.sqrt((torch.where(full, m - mean, torch.zeros_like(m)) ** 2).sum(1, keepdim=True) / n)
    x = torch.where(full & (sd > 0), mean + (v - mean) / torch.where(sd > 0, sd, torch.ones_like(sd)), mean)
    x = x[:, None, :]
    for k in ("conv1", "conv2", "conv3"):
        x = torch.relu(_conv(x, w[k + ".w"], w[k + ".b"]))
        x = torch.maximum(x[:, :, 0::2], x[:, :, 1::2])
    x = torch.relu(x.reshape(x.shape[0], -1) @ w["fc1.w"].T + w["fc1.b"])
    return (x @ w["fc2.w"].T + w["fc2.b"]).reshape(-1)


def _scores(case, t, f, p, t0, w):
    """Scores of one star in 64 bits."""
    tau, x, ref = _quantised(t, f, t0)
    sigma = torch.sqrt((x * x).mean())
    out = torch.empty(len(p), dtype=torch.float64, device=p.device)
    for a, s, c in _folds(tau, x, p, case["nbins"], 1 << (26 if case["scorer"] == "box" else 25)):
        if case["scorer"] == "box":
            out[a:a + len(s)] = _box(s, c, case["w_max"], sigma)
        else:
            out[a:a + len(s)] = torch.sigmoid(_logits(ref + s / c.clamp(min=1), c, w))
    return out


def _star(score):
    mean = score.mean()
    sd = torch.sqrt(((score - mean) ** 2).mean())
    return torch.stack([(score.max() - mean) / sd, mean, sd])


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    M = 0xFFFFFFFF
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
        p0, p1 = 0xD2511F53 * c0, 0xCD9E8D57 * c2
        c0, c1, c2, c3 = ((p1 >> 32) & M) ^ c1 ^ k0, p1 & M, ((p0 >> 32) & M) ^ c3 ^ k1, p0 & M
    return c0, c1, c2, c3


def _synth(case, seed):
    sp = dict(g.TRAINING_SET, n_cadences=case["n_cad"])
    n, nb, nc = case["n"], case["nbins"], case["n_cad"]
    dev, k0, k1 = "cuda", seed & 0xFFFFFFFF, seed >> 32
    j = torch.arange(n, device=dev)
    zero = torch.zeros_like(j)
    unit = lambda v: (v >> 8).double() / 16777216.0  # noqa: E731
    a = [unit(v) for v in _philox(j, zero, zero, zero + 0xFFFFFFFF, k0, k1)]
    b = [unit(v) for v in _philox(j, zero + 1, zero, zero + 0xFFFFFFFF, k0, k1)]
    logu = lambda u, lo, hi: torch.exp(math.log(lo) + u * math.log(hi / lo))  # noqa: E731
    kind = torch.where(j % 2 == 1, 1 + (j // 2) % 3, zero)
    sigma = logu(a[0], sp["sigma_min"], sp["sigma_max"])
    period = sp["p_min"] + a[1] * (sp["p_max"] - sp["p_min"])
    epoch = a[2] * period
    dur = (sp["dur_min_h"] + a[3] * (sp["dur_max_h"] - sp["dur_min_h"])) / 24.0
    depth = logu(b[0], sp["depth_min"], sp["depth_max"])
    depth2 = depth * (0.2 + 0.8 * b[1])
    amp = logu(b[2], sp["depth_min"], sp["depth_max"])
    df = (2.0 * b[3] - 1.0) * sp["drift_bins"] / (256.0 * (nc * sp["cadence"]))
    fold = 1.0 / (1.0 / period + df)
    i = torch.arange(nc, device=dev)
    t = i.double() * sp["cadence"]
    tau = torch.round(t * 16777216.0).to(torch.int64)
    folded = torch.empty((n, nb), dtype=torch.float64, device=dev)
    std = torch.empty(n, dtype=torch.float64, device=dev)
    q = (nc + 3) // 4
    step = max(1, (1 << 25) // nc)
    for lo in range(0, n, step):
        e = slice(lo, min(n, lo + step))
        jj = j[e][:, None].expand(-1, q)
        m = torch.arange(q, device=dev)[None, :].expand(len(jj), -1)
        r = _philox(jj, m, torch.ones_like(m), torch.zeros_like(m), k0, k1)
        z = torch.empty((len(jj), q, 4), dtype=torch.float64, device=dev)
        for h in range(2):
            rad = torch.sqrt(-2.0 * torch.log(1.0 - unit(r[2 * h])))
            z[:, :, 2 * h] = rad * torch.cos(2 * math.pi * unit(r[2 * h + 1]))
            z[:, :, 2 * h + 1] = rad * torch.sin(2 * math.pi * unit(r[2 * h + 1]))
        col = lambda v: v[e][:, None]  # noqa: E731
        x = col(sigma) * z.reshape(len(jj), -1)[:, :nc]

        def inside(centre):
            P = col(period)
            d = torch.fmod(t[None, :] - centre + 0.5 * P, P)
            d = torch.where(d < 0, d + P, d) - 0.5 * P
            return d.abs() < 0.5 * col(dur)

        box = inside(col(epoch)).double()
        x = x - torch.where((col(kind) == 0) | (col(kind) == 3), box * col(depth), torch.zeros_like(x))
        box = inside(col(epoch) + 0.5 * col(period)).double()
        x = x - torch.where(col(kind) == 3, box * col(depth2), torch.zeros_like(x))
        wave = col(amp) * torch.sin(2 * math.pi * ((t[None, :] - col(epoch)) / col(period)))
        x = x + torch.where(col(kind) == 2, wave, torch.zeros_like(x))
        std[e] = torch.sqrt(((x - x.mean(1, keepdim=True)) ** 2).mean(1))
        bins = _bins(tau, fold[e], nb) + nb * torch.arange(len(jj), device=dev)[:, None]
        s = torch.zeros(len(jj) * nb, dtype=torch.float64, device=dev).scatter_add_(0, bins.reshape(-1), x.reshape(-1))
        c = torch.zeros_like(s).scatter_add_(0, bins.reshape(-1), torch.ones_like(x).reshape(-1))
        folded[e] = torch.where(c > 0, 1.0 + s / c, torch.full_like(s, math.nan)).view(-1, nb)
    return {"folded": folded, "counts": None, "label": (kind == 0).double(), "period": fold, "flux_std": std}


def _spline_basis(t, knots):
    """Cubic B-splines at t by the Cox-de Boor recursion; the last knot belongs to the last interval."""
    k = torch.tensor(knots, dtype=torch.float64, device=t.device)
    B = ((k[None, :-1] <= t[:, None]) & (t[:, None] < k[None, 1:])).double()
    B[t == k[-1], len(knots) - 5] = 1.0
    for d in range(1, 4):
        n = len(knots) - 1 - d
        dl, dr = k[d:d + n] - k[:n], k[d + 1:d + 1 + n] - k[1:1 + n]
        left = torch.where(dl > 0, (t[:, None] - k[None, :n]) / torch.where(dl > 0, dl, torch.ones_like(dl)), 0.0)
        right = torch.where(dr > 0, (k[None, d + 1:d + 1 + n] - t[:, None]) / torch.where(dr > 0, dr, torch.ones_like(dr)), 0.0)
        B = left * B[:, :n] + right * B[:, 1:n + 1]
    return B


def _spline_fit(t, f, free, spacing):
    """(BIC, trend) of the clipped least-squares spline of one segment, or None."""
    t0, t1 = float(t[0]), float(t[-1])
    inner, j = [], 1
    while t0 + spacing * j < t1:
        inner.append(t0 + spacing * j)
        j += 1
    B = _spline_basis(t, [t0] * 4 + inner + [t1] * 4)
    p = B.shape[1]
    if p > len(t):
        return None
    D = torch.zeros((p - 2, p), dtype=torch.float64, device=t.device)
    r = torch.arange(p - 2, device=t.device)
    D[r, r], D[r, r + 1], D[r, r + 2] = 1.0, -2.0, 1.0
    used = free.clone()
    for it in range(10):
        n = int(used.sum())
        if n < p:
            return None
        Bu = B * used[:, None]
        G = Bu.T @ B
        c = torch.linalg.solve(G + 1e-9 * torch.trace(G) / p * (D.T @ D), Bu.T @ f)
        trend = B @ c
        res = f - trend
        rss = float((res[used] ** 2).sum())
        thr = max(3.0 * math.sqrt(rss / n), 1e-9 * math.sqrt(float((f[used] ** 2).mean())))
        nxt = free & (res.abs() <= thr)
        if it == 9 or torch.equal(nxt, used):
            break
        used = nxt
    return (n * math.log(rss / n) + p * math.log(n) if rss > 0 else -math.inf), trend


def _detrended(t, f, mask):
    f = f.double()
    sd = torch.sqrt(((f - f.mean()) ** 2).mean())
    cut = (t[1:] - t[:-1] > 30 * 0.020428) | ((f[1:] - f[:-1]).abs() > 5.0 * sd)
    edges = [0] + (torch.nonzero(cut).reshape(-1) + 1).tolist() + [len(t)]
    ts, fs = [], []
    for a, b in zip(edges[:-1], edges[1:]):
        if b - a <= 60:
            continue
        best = None
        for sp in SPACINGS:
            r = _spline_fit(t[a:b], f[a:b], mask[a:b] == 0, sp)
            if r is not None and (best is None or r[0] < best[0]):
                best = r
        if best is not None:
            ts.append(t[a + 30:b - 30])
            fs.append((f[a:b] / best[1])[30:-30])
    return {"times": torch.cat(ts), "flux": torch.cat(fs), "segment": None}


def exact(case, seed):
    st, kind = prepare(case, seed), case["kind"]
    w = {n: v.double() for n, v in st["w"].items()} if "w" in st else None
    if kind == "search":
        score = _scores(case, st["t"], st["f"], st["p"], st["t0"], w)
        return {"score": score, "best_index": None, "best_score": score.max().reshape(1),
                "star": {"sde_mean_sd": _star(score)[None, :], "best_index": None, "best_score": None, "n_peaks": None}}
    if kind == "batch":
        scores, a, b = [], 0, 0
        for n, m in zip(st["lens"], st["grids"]):
            scores.append(_scores(case, st["t"][a:a + n], st["f"][a:a + n], st["p"][b:b + m], 0.0, w))
            a, b = a + n, b + m
        return {"score": torch.cat(scores), "best_index": None, "best_score": torch.stack([s.max() for s in scores]),
                "star": {"sde_mean_sd": torch.stack([_star(s) for s in scores]), "best_index": None, "best_score": None,
                         "n_peaks": None}}
    if kind == "fold":
        tau, x, ref = _quantised(st["t"], st["f"], st["t0"])
        out = [torch.where(c > 0, ref + s / c.clamp(min=1), torch.full_like(s, math.nan))
               for _, s, c in _folds(tau, x, st["p"], case["nbins"])]
        return {"folded": torch.cat(out), "counts": None}
    if kind == "equal":
        tau, x, ref = _quantised(st["t"], st["f"], st["t0"])
        n, nb, out = len(tau), case["nbins"], []
        u = n * torch.arange(nb + 1, device="cuda", dtype=torch.float64)  # boundaries in units of 1/nb sample
        for _, s, c in _folds(tau, x, st["p"], case["nfine"]):
            C, S = c.cumsum(1) * nb, s.cumsum(1)
            f = torch.searchsorted(C, u.expand(len(C), -1).contiguous()).clamp(max=case["nfine"] - 1)
            cf, sf = c.gather(1, f) * nb, s.gather(1, f)
            G = S.gather(1, f) - sf + sf * (u - (C.gather(1, f) - cf)) / cf.clamp(min=1)
            G[:, 0] = 0.0
            out.append(ref + (G[:, 1:] - G[:, :-1]) * (nb / n))
        return {"folded": torch.cat(out)}
    if kind == "score_box":
        out = []
        for a in range(0, case["n"], 16384):
            c = st["counts"][a:a + 16384].double()
            m = st["prof"][a:a + 16384].double()
            ref = (m * c).sum(1, keepdim=True) / c.sum(1, keepdim=True)
            out.append(_box((m - ref) * c, c, case["w_max"], 1.0))
        return {"score": torch.cat(out), "best_s": None, "best_w": None}
    if kind == "score_cnn":
        out = [torch.sigmoid(_logits(st["prof"][a:a + 8192].double(), st["counts"][a:a + 8192], w))
               for a in range(0, case["n"], 8192)]
        return {"score": torch.cat(out)}
    if kind == "train":
        for v in w.values():
            v.requires_grad_(True)
        y = st["label"].double()
        z = _logits(st["prof"].double(), st["counts"], w)
        loss = (z.clamp(min=0) - z * y + torch.log1p(torch.exp(-z.abs()))).mean()
        loss.backward()
        grads, new, step = {n: v.grad for n, v in w.items()}, {}, st["step"] + 1
        for n in w:
            m = 0.9 * st["m"][n].double() + 0.1 * grads[n]
            v = 0.999 * st["v"][n].double() + 0.001 * grads[n] ** 2
            new[n] = (w[n] - 1e-3 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)).detach()
        return {"logit": z.detach(), "loss": loss.detach().reshape(1), "grads": grads, "weights": new}
    if kind == "synth":
        return _synth(case, int(seed))
    return _detrended(st["t"], st["f"], st["mask"])
