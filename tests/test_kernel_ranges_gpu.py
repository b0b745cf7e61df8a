"""Ranges beyond the usual ones: long generated curves, flux with outliers or that is no number, resonant and
irregular times, wide profiles, large scales, and the workspace. Times are compared on the same GPU in the same
process, with room for noise."""
import numpy as np
import pytest
import torch

import lcsynth
import oracle

pytestmark = pytest.mark.gpu
CADENCE = 29.4 / 1440.0


@pytest.fixture(scope="module")
def ctx():
    import paper_2312_02063_gb300 as g
    c = g.Context(0)
    yield c
    c.close()


def _dev(ctx, a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(ctx.device)


def _ms(ctx, call, reps=5):
    """Least time of a call, after two warm-up calls."""
    for _ in range(2):
        call()
    ctx.sync()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = float("inf")
    for _ in range(reps):
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


# ---------------------------------------------------------------- generated profiles

def test_flux_std_of_a_long_sinusoid(ctx):
    """2^27 cadences whose squares sum to more than 64 bits of the integers they are added as. The
    expected value is that of whole cycles; a part of one among 10^5 changes it by 1e-6."""
    import paper_2312_02063_gb300 as g
    amp, sigma = 0.0019, 1e-6
    sp = dict(g.TRAINING_SET, n_cadences=1 << 27, cadence=1 / 1440.0, depth_min=amp, depth_max=amp, sigma_min=sigma,
              sigma_max=sigma)
    _, counts, _, _, std = g.gpfc_synth_profiles(ctx, 5, 3, 1, 256, sp, want_std=True)  # curve 3: a sinusoid
    ctx.sync()
    assert int(counts.sum().item()) == 1 << 27
    assert abs(float(std[0]) / (amp * amp / 2 + sigma * sigma) ** 0.5 - 1.0) <= 1e-5


@pytest.mark.parametrize("n_cad,nbins", [(300, 256), (5003, 37), (131073, 200)])
def test_flux_std_does_not_depend_on_the_batch(ctx, n_cad, nbins):
    import paper_2312_02063_gb300 as g
    sp = dict(lcsynth.TRAINING_SET, n_cadences=n_cad)
    many = g.gpfc_synth_profiles(ctx, 9, 40, 640, nbins, sp, want_std=True)[4]
    for j in (0, 1, 3, 639):
        one = g.gpfc_synth_profiles(ctx, 9, 40 + j, 1, nbins, sp, want_std=True)[4]
        ctx.sync()
        assert abs(float(one[0]) / float(many[j]) - 1.0) <= 2.0 ** -23


# noise of a few parts in ten, deep signals on quiet stars, few samples a bin. Off by at most half a
# unit in the last place of a mean between 1 and 2 and one rounding of the largest sample
@pytest.mark.parametrize("sigma,depth,n_cad", [((0.05, 0.3), (3e-5, 2e-3), 20000), ((1e-7, 1e-6), (0.3, 0.9), 400),
                                               ((1e-4, 1e-3), (0.3, 0.9), 6000)])
def test_generated_profiles_of_wide_ranges(ctx, sigma, depth, n_cad):
    import paper_2312_02063_gb300 as g
    sp = dict(lcsynth.TRAINING_SET, n_cadences=n_cad, sigma_min=sigma[0], sigma_max=sigma[1], depth_min=depth[0],
              depth_max=depth[1])
    f, c, _, per, std = g.gpfc_synth_profiles(ctx, 31, 0, 36, 256, sp, want_period=True, want_std=True)
    ctx.sync()
    f, c, per, std = (x.cpu().numpy() for x in (f, c, per, std))
    err = []
    for j in range(36):
        t, flux, _, P = lcsynth.training_light_curve(31, j, sp)
        assert per[j] == P
        b = oracle.bins(oracle.quantise_times(t, 0.0), oracle.quantise_periods(np.array([P])), 256)[0]
        cnt = np.bincount(b, minlength=256)
        np.testing.assert_array_equal(c[j], cnt)
        nz = cnt > 0
        mean = 1.0 + np.bincount(b, weights=flux - 1.0, minlength=256)[nz] / cnt[nz]
        e = np.abs(f[j][nz].astype(np.float64) - mean)
        assert e.max() <= 2.0 ** -24 + 2.0 ** -25 * np.abs(flux - 1.0).max(), j
        err.append(e)
        assert abs(std[j] / np.std(flux) - 1.0) <= 2.0 ** -22
    assert np.sqrt((np.concatenate(err) ** 2).mean()) <= 2.0 ** -23 / 12 ** 0.5


# ---------------------------------------------------------------- flux

@pytest.mark.parametrize("nbins", [256, 300, 512])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("width", [1.0, 0.5, 0.125])
def test_counts_with_a_flux_that_is_no_number(ctx, nbins, bad, width):
    """The counts stay exact (phases in all of a period and in parts of it, some 128 samples a bin and
    segment), the means are no numbers, and the scores are those of the two-word fold."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(1)
    n = 65000
    t = np.arange(n) // 128 + (np.arange(n) % 128) / 128.0 * width + 1e-4
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    f[77] = bad
    p = np.r_[1.0, 0.5, rng.uniform(0.3, 1.0, 300)]
    args = [_dev(ctx, x) for x in (t, f, p)]
    try:
        if nbins in (256, 512):
            ctx.set_fold_config(**_one_word(g, 3))
        folded, counts = g.gpfc_fold(ctx, *args, nbins, 0.0)
        score, _, _ = g.gpfc_search(ctx, *args, nbins, 0.0, g.SCORER_BOX, 1, 20, 0.0)
        ctx.set_fold_config(warps=1, layout=g.LAYOUT_RED32)
        folded2, counts2 = g.gpfc_fold(ctx, *args, nbins, 0.0)
        score2, _, _ = g.gpfc_search(ctx, *args, nbins, 0.0, g.SCORER_BOX, 1, 20, 0.0)
    finally:
        ctx.reset_fold_config()
    ctx.sync()
    assert torch.equal(counts, counts2)
    assert torch.equal(torch.isfinite(folded), torch.isfinite(folded2)) and not torch.isfinite(folded).any()
    assert torch.equal(torch.nan_to_num(score, 7.0), torch.nan_to_num(score2, 7.0))
    _, cnt_o, _ = oracle.fold(t, np.ones(n, np.float32), p[:6], nbins, 0.0)
    np.testing.assert_array_equal(counts[:6].cpu().numpy(), cnt_o)


# an outlier far above a flux about zero, or above its level: the FP32 sums; none, one within the level or a
# normal spread about zero: 31 bits of the largest value, which are the more exact there
@pytest.mark.parametrize("level,outlier,fp32", [(0.0, 1e6, True), (1.0, 1e6, True), (0.0, 1.0, True), (0.0, 0.0, False),
                                                (1.0, 0.0, False), (1.0, 1.0, False), (1e5, 1e4, False)])
@pytest.mark.parametrize("nbins", [64, 200])
def test_fold_below_256_bins_with_an_outlier(ctx, level, outlier, fp32, nbins):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(2)
    n = 20000
    t = np.arange(n) * CADENCE
    f = (level + rng.normal(0.0, 3e-4 * max(level, 1.0), n)).astype(np.float32)
    f[5] += np.float32(outlier)
    p = rng.uniform(0.2, 1.0, 50)
    args = [_dev(ctx, x) for x in (t, f, p)]
    a, ca = g.gpfc_fold(ctx, *args, nbins, 0.0)
    ctx.set_fold_config(layout=1)
    try:
        b, cb = g.gpfc_fold(ctx, *args, nbins, 0.0)
    finally:
        ctx.reset_fold_config()
    ctx.sync()
    assert torch.equal(ca, cb)
    if fp32:
        assert torch.equal(torch.nan_to_num(a, 7.0), torch.nan_to_num(b, 7.0))
        return
    mean_o, cnt_o, _ = oracle.fold(t, f, p, nbins, 0.0)
    nz = cnt_o > 0
    rms = [np.sqrt(((x.cpu().numpy().astype(np.float64)[nz] - mean_o[nz]) ** 2).mean()) for x in (a, b)]
    assert rms[0] <= rms[1] * (1.0 + 1e-3)


# ---------------------------------------------------------------- the one-word fold's range

def _times(kind, n, rng):
    t = np.arange(n) * CADENCE
    if kind == "gaps":
        t = t + 3.3 * (np.arange(n) // 911)
    elif kind == "nights":
        t = np.arange(n) // 1200 + (np.arange(n) % 1200) / 3600.0
    elif kind == "unsorted":
        t = rng.uniform(0.0, 900.0, n)
    elif kind == "random":  # no cadence: the smallest step says nothing about the others
        t = np.sort(rng.uniform(0.0, n * CADENCE, n))
    elif kind == "equal":  # every sample in one bin of every period
        t = np.full(n, 7.25)
    elif kind == "barycentric":
        t = t + 200.0 / 86400.0 * np.sin(2 * np.pi * t / 372.5)
    return t


def _one_word(g, groups):
    """The one-word fold by its own shape, with that many groups of 32 periods a block."""
    return dict(warps=groups, layout=g.LAYOUT_RED32, tile=2048, blocks_per_sm=1, streams=1)


# lengths about the tile (256 to 2,048), the segments (1 to 8 tiles), the chunk (65,520) and the groups of 16;
# periods about the group (32) and the block; a fine grid about twelve and a half cadences, whose groups
# fail their checks and go on with shorter segments
@pytest.mark.parametrize("n,kind,n_periods,nbins,groups", [
    (1, "regular", 1, 256, 1), (15, "regular", 33, 256, 2), (17, "unsorted", 31, 512, 1), (300, "gaps", 193, 256, 6),
    (2047, "regular", 200, 256, 6), (2049, "gaps", 64, 256, 2), (4096, "equal", 40, 256, 3), (3000, "random", 700, 512, 3),
    (20000, "barycentric", 500, 256, 4), (32769, "gaps", 193, 256, 5), (65519, "regular", 96, 256, 3),
    (65521, "gaps", 192, 256, 6), (70001, "unsorted", 65, 512, 2), (140000, "nights", 200, 256, 6),
    (40000, "equal", 33, 512, 3), (200000, "random", 64, 256, 2)])
def test_one_word_fold_equals_two_words(ctx, n, kind, n_periods, nbins, groups):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(n + nbins)
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    p = np.r_[np.linspace(12.45, 12.55, n_periods // 2) * CADENCE, rng.uniform(0.05, 1.0, n_periods - n_periods // 2)]
    args = [_dev(ctx, x) for x in (_times(kind, n, rng), f, p)]
    try:
        ctx.set_fold_config(**_one_word(g, groups))
        one = g.gpfc_fold(ctx, *args, nbins, 0.0)
        assert ctx.last_fold_plan()["warps"] == groups and ctx.last_fold_plan()["streams"] == 1
        ctx.set_fold_config(warps=1, layout=g.LAYOUT_RED32)
        two = g.gpfc_fold(ctx, *args, nbins, 0.0)
    finally:
        ctx.reset_fold_config()
    ctx.sync()
    assert torch.equal(one[1], two[1])
    assert torch.equal(torch.nan_to_num(one[0], 7.0), torch.nan_to_num(two[0], 7.0))


def test_one_word_fold_of_hard_periods_takes_at_most_a_second_turn(ctx):
    """Periods all within 10^-4 of seven cadences (every sample in seven bins), and times without a cadence,
    against periods that spread the samples: no sample is folded more than twice, but for a failed segment."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(5)
    f = (1.0 + rng.normal(0.0, 3e-4, 65000)).astype(np.float32)
    easy, narrow = np.linspace(24.5, 4900.0, 29184) * CADENCE, np.linspace(6.999, 7.001, 29184) * CADENCE
    t = []
    ctx.set_fold_config(**_one_word(g, 6))
    try:
        for kind, p in (("regular", easy), ("regular", narrow), ("random", easy)):
            args = [_dev(ctx, x) for x in (_times(kind, 65000, rng), f, p)]
            t.append(_ms(ctx, lambda: g.gpfc_fold(ctx, *args, 256, 0.0)))  # noqa: B023
    finally:
        ctx.reset_fold_config()
    assert t[1] <= 2.2 * t[0] and t[2] <= 1.2 * t[0]


# below 256 bins with many groups a multiprocessor (5 groups have no instance of their own)
@pytest.mark.parametrize("n_periods,nbins", [(24000, 64), (24000, 100), (60011, 32)])
def test_fold_below_256_bins_of_long_grids(ctx, n_periods, nbins):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(nbins)
    n = 24001
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    args = [_dev(ctx, x) for x in (_times("gaps", n, rng), f, rng.uniform(0.05, 1.0, n_periods))]
    a, ca = g.gpfc_fold(ctx, *args, nbins, 0.0)
    ctx.set_fold_config(layout=1)
    try:
        b, cb = g.gpfc_fold(ctx, *args, nbins, 0.0)
    finally:
        ctx.reset_fold_config()
    ctx.sync()
    assert torch.equal(ca, cb) and torch.equal(torch.isfinite(a), torch.isfinite(b))
    assert not torch.equal(torch.nan_to_num(a, 7.0), torch.nan_to_num(b, 7.0))  # (another sum: the one-word fold ran)
    assert float((torch.nan_to_num(a, 1.0) - torch.nan_to_num(b, 1.0)).abs().max()) <= 2.0 ** -22


def test_plans_of_the_one_word_fold_name_it(ctx):
    """The plan given out, set by hand, is the same fold of the same shape; so is the autotuner's."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(3)
    n = 62000
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    args = [_dev(ctx, x) for x in (_times("gaps", n, rng), f, np.linspace(0.2, 1.0, 30000))]
    for two_words in (False, True):
        p = args[2][:2000] if two_words else args[2]
        try:
            a = g.gpfc_fold(ctx, args[0], args[1], p, 256, 0.0)
            plan = ctx.last_fold_plan()
            assert (plan["streams"] == 1) != two_words
            ctx.set_fold_config(**plan)
            b = g.gpfc_fold(ctx, args[0], args[1], p, 256, 0.0)
            assert ctx.last_fold_plan() == plan
        finally:
            ctx.reset_fold_config()
        ctx.sync()
        assert torch.equal(a[1], b[1]) and torch.equal(torch.nan_to_num(a[0], 7.0), torch.nan_to_num(b[0], 7.0))
    try:
        cfg = g.gpfc_autotune(ctx, *args, 256, g.SCORER_BOX, 1, 40, 0.0)
        ref, _, _ = g.gpfc_search(ctx, *args, 256, 0.0, g.SCORER_BOX, 1, 40, 0.0)
        plan = ctx.last_fold_plan()
        ctx.set_autotune(-1)
        ctx.set_fold_config(**cfg)
        sc, _, _ = g.gpfc_search(ctx, *args, 256, 0.0, g.SCORER_BOX, 1, 40, 0.0)
        assert ctx.last_fold_plan() == plan
    finally:
        ctx.reset_fold_config()
        ctx.set_autotune(-1)
        ctx.set_autotune(1)
    ctx.sync()
    assert torch.equal(ref, sc)


# the automatic fold against the two-word fold's automatic shape: no slower, wherever the periods lie
# about the cadence, whatever the times, short and long (a fifth for noise)
@pytest.mark.parametrize("n,kind,n_periods,nbins", [
    (100, "regular", 40, 256), (1000, "regular", 60000, 256), (3000, "random", 20000, 256), (3000, "random", 20000, 512),
    (20000, "gaps", 10000, 256), (20000, "gaps", 10000, 300), (65000, "gaps", 1000, 256), (65000, "gaps", 10000, 512),
    (65000, "gaps", 30000, 256), (65000, "random", 30000, 256), (65000, "barycentric", 30000, 512), (5000, "gaps", 20000, 700)])
def test_automatic_fold_is_no_slower_than_two_words(ctx, n, kind, n_periods, nbins):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(n)
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    args = [_dev(ctx, x) for x in (_times(kind, n, rng), f, 1.0 / np.linspace(1.0, 5.0, n_periods))]
    call = lambda: g.gpfc_fold(ctx, *args, nbins, 0.0)  # noqa: E731
    auto = _ms(ctx, call)
    per_sm = -(-n_periods // (32 * ctx.num_sms))
    ctx.set_fold_config(warps=max(1, min(per_sm, ctx.fold_max_warps(nbins, 3))), layout=g.LAYOUT_RED32)
    try:
        two = _ms(ctx, call)
    finally:
        ctx.reset_fold_config()
    assert auto <= 1.2 * two


@pytest.mark.parametrize("n,n_periods,nbins", [(100, 60000, 64), (1000, 60000, 32), (2000, 20000, 200), (24000, 60000, 100),
                                               (65000, 10000, 64), (300, 3000, 128)])
def test_automatic_fold_below_256_bins_is_no_slower_than_fp32(ctx, n, n_periods, nbins):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(n)
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    args = [_dev(ctx, x) for x in (_times("gaps", n, rng), f, 1.0 / np.linspace(1.0, 5.0, n_periods))]
    call = lambda: g.gpfc_fold(ctx, *args, nbins, 0.0)  # noqa: E731
    auto = _ms(ctx, call)
    ctx.set_fold_config(layout=1)
    try:
        fp32 = _ms(ctx, call)
    finally:
        ctx.reset_fold_config()
    assert auto <= 1.2 * fp32


# ---------------------------------------------------------------- box scorer, decision

def test_box_scorer_of_wide_smooth_profiles(ctx):
    """A smooth profile of thousands of bins costs what noise does."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(1)
    x = np.arange(4096) / 4096
    smooth = 1.0 + 1e-3 * np.sin(2 * np.pi * (x[None] + rng.uniform(0, 1, (600, 1))))
    noise = 1.0 + rng.normal(0, 1e-4, (600, 4096))
    counts = _dev(ctx, np.full((600, 4096), 40, np.int32))
    t = [_ms(ctx, lambda p=_dev(ctx, p.astype(np.float32)): g.gpfc_score_box(ctx, p, counts, 1, 1720, 1e-4))
         for p in (smooth, noise)]
    assert t[0] <= 1.25 * t[1]


@pytest.mark.parametrize("scale", [1e-25, 1.0, 1e12])
def test_box_scores_of_any_scale_are_the_same_on_every_path(ctx, scale):
    """The separate scorer against the one-kernel search, whose comparisons it promises, also where their
    products leave the FP32 range."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(4)
    n = 3000
    f = (scale * (1.0 + rng.normal(0.0, 0.3, n))).astype(np.float32)
    args = [_dev(ctx, x) for x in (_times("gaps", n, rng), f, rng.uniform(0.2, 1.0, 300))]
    out = []
    try:
        ctx.set_fold_config(warps=2, layout=1)
        for path in (g.BOX_WARP, g.BOX_FUSED):
            ctx.set_box_path(path)
            out.append(g.gpfc_search(ctx, *args, 256, 0.0, g.SCORER_BOX, 1, 60, scale * 0.3)[0])
    finally:
        ctx.set_box_path(g.BOX_AUTO)
        ctx.reset_fold_config()
    ctx.sync()
    assert torch.equal(torch.nan_to_num(out[0], 7.0), torch.nan_to_num(out[1], 7.0))


# boxes that start with empty bins tie with the next start's, but not across a block of eight starts or the end
@pytest.mark.parametrize("n,nbins", [(20, 100), (60, 256), (150, 256), (150, 300), (400, 301), (90, 64)])
def test_box_scores_of_sparse_profiles_are_the_same_on_every_path(ctx, n, nbins):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(n)
    f = (1.0 + rng.normal(0.0, 1e-3, n)).astype(np.float32)
    args = [_dev(ctx, x) for x in (_times("random", n, rng), f, rng.uniform(0.2, 1.0, 2000))]
    out = []
    try:
        ctx.set_fold_config(warps=2, layout=1)
        for path in (g.BOX_WARP, g.BOX_EPILOGUE):
            ctx.set_box_path(path)
            out.append(g.gpfc_search(ctx, *args, nbins, 0.0, g.SCORER_BOX, 1, nbins // 2, 1e-3)[0])
    finally:
        ctx.set_box_path(g.BOX_AUTO)
        ctx.reset_fold_config()
    ctx.sync()
    assert torch.equal(torch.nan_to_num(out[0], 7.0), torch.nan_to_num(out[1], 7.0))


def test_box_scorer_of_sparse_profiles(ctx):
    """A profile with every second bin empty costs no more than a full one."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(2)
    t = []
    for density in (0.6, 40.0):
        c = rng.poisson(density, (1000, 512)).astype(np.int32)
        p = np.where(c > 0, 1.0 + rng.normal(0, 1e-4, c.shape), np.nan).astype(np.float32)
        args = [_dev(ctx, p), _dev(ctx, c)]
        t.append(_ms(ctx, lambda: g.gpfc_score_box(ctx, *args, 1, 128, 1e-4), reps=20))  # noqa: B023
    assert t[0] <= 1.4 * t[1]


def test_decision_of_several_stars_takes_no_longer_than_of_many(ctx):
    """19 stars of 16,384 periods: a block each, not clusters that take turns."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(6)
    n = 16384

    def of(stars):
        s = _dev(ctx, rng.normal(0, 1, stars * n).astype(np.float32))
        p = _dev(ctx, np.tile(np.linspace(0.2, 30.0, n), stars))
        off = _dev(ctx, (np.arange(stars + 1) * n).astype(np.int64))
        return _ms(ctx, lambda: g.gpfc_peaks(ctx, s, p, off, max_peaks=4), reps=20)
    assert of(19) <= 1.25 * of(60)


# ---------------------------------------------------------------- detrending

def test_detrending_workspace_and_spacings_in_groups(ctx):
    """1.2 million samples with eight spacings: the spacings go through in groups. The halves, each in one
    group, give the same bits (no flux gap; the cut lies at a time gap), and the workspace stays near 1 GiB."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(8)
    n = 1200000
    t = np.arange(n) * CADENCE + 4.0 * (np.arange(n) // 1500)
    f = _dev(ctx, (1.0 + 1e-3 * np.sin(t / 2.0) + rng.normal(0, 2e-4, n)).astype(np.float32))
    t = _dev(ctx, t)
    kw = dict(edge=5, flux_gap_sigma=1e9, spacings=[0.4, 0.5, 0.7, 1.0, 1.5, 2.0, 3.0, 5.0], max_iter=3)
    fresh = g.Context(0)
    try:
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        whole = g.gpfc_detrend(fresh, t, f, None, **kw)
        fresh.sync()
        held = before - torch.cuda.mem_get_info()[0]
        whole = [x.clone() for x in whole]
        assert held <= 1.5 * 2 ** 30  # (1 GiB, an eighth more, 44 bytes a sample and the outputs)
        h = n // 2
        parts = [g.gpfc_detrend(fresh, t[a:a + h].contiguous(), f[a:a + h].contiguous(), None, **kw) for a in (0, h)]
        fresh.sync()
        for i in range(2):
            assert torch.equal(whole[i], torch.cat([p[i] for p in parts]))
    finally:
        fresh.close()


def test_detrending_of_a_segment_longer_than_a_tile_of_intervals(ctx):
    """One segment with 571 and 142 knot intervals (a block sums 256 at a time) against the oracle."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(9)
    n = 7000
    t = np.arange(n) * CADENCE
    f = (1.0 + 1e-3 * np.sin(t / 3.0) + 3e-4 * np.sin(t * 4.0) + rng.normal(0, 1e-4, n)).astype(np.float32)
    to, fo, _ = g.gpfc_detrend(ctx, _dev(ctx, t), _dev(ctx, f), None, spacings=[0.25, 1.0])
    ctx.sync()
    r = oracle.detrend(t, f, None, spacings=(0.25, 1.0))
    np.testing.assert_array_equal(to.cpu().numpy(), r["times"])
    assert (np.abs(fo.cpu().numpy().astype(np.float64) / r["flux"] - 1.0)).max() <= 2e-7
