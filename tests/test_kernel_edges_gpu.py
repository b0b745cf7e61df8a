"""Sizes at which the kernels change their split, tile or path: each against the FP64 oracle, the
general path or the same work in another shape."""
import numpy as np
import pytest
import torch

import lcsynth
import oracle

pytestmark = pytest.mark.gpu
CADENCE = 29.4 / 1440.0
MEAN_RTOL = 1e-6   # bin means, as for every fold
BOX_RTOL = 1e-5    # box-SNR, as for every box search
FLUX_RTOL = 2e-7   # detrended flux, as for every detrending


@pytest.fixture(scope="module")
def ctx():
    import paper_2312_02063_gb300 as g
    c = g.Context(0)
    yield c
    c.close()


def _dev(ctx, a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(ctx.device)


# below 256 bins: about the tile (2,048), the segments (a mean load of half a word's 256 counts), the
# chunk (65,520), the groups of 32 periods a block takes (1, 2, 3, 6; 4 and 5 in a last chunk) and the
# fewest bins (32)
@pytest.mark.parametrize("n,kind,n_periods,nbins", [
    (1, "regular", 1, 32), (17, "unsorted", 33, 31), (2047, "gaps", 65, 33), (2049, "regular", 193, 64),
    (3000, "equal", 40, 128), (5001, "unsorted", 97, 200), (40000, "gaps", 34, 255), (30000, "regular", 70, 32),
    (65521, "gaps", 33, 200), (140000, "unsorted", 20, 48), (300, "regular", 29184 + 19456, 64),
    (300, "unsorted", 29184 + 24000, 100)])
def test_fold_below_256_bins(ctx, n, kind, n_periods, nbins):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(n + nbins)
    t = np.arange(n) * CADENCE
    if kind == "gaps":
        t = t + 3.3 * (np.arange(n) // 911)
    elif kind == "unsorted":
        t = rng.uniform(0.0, 900.0, n)
    elif kind == "equal":  # every sample in one bin of every period
        t = np.full(n, 7.25)
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    p = rng.uniform(0.2, 1.0, n_periods)
    if n_periods > 2:
        p[1] = 10 * CADENCE
    td, fd, pd = _dev(ctx, t), _dev(ctx, f), _dev(ctx, p)
    folded, counts = g.gpfc_fold(ctx, td, fd, pd, nbins, 0.0)
    ctx.set_fold_config(layout=1)  # the general path
    try:
        folded_e, counts_e = g.gpfc_fold(ctx, td, fd, pd, nbins, 0.0)
    finally:
        ctx.reset_fold_config()
    ctx.sync()
    fo, co = folded.cpu().numpy(), counts.cpu().numpy()
    np.testing.assert_array_equal(co, counts_e.cpu().numpy())
    np.testing.assert_array_equal(np.isnan(fo), co == 0)
    nz = co > 0
    fe = folded_e.cpu().numpy()
    assert np.all(np.abs(fo[nz] - fe[nz]) <= 2 * MEAN_RTOL * np.abs(fe[nz]))
    idx = np.unique(np.r_[0:min(n_periods, 12), n_periods - 1])
    mean_o, cnt_o, _ = oracle.fold(t, f, p[idx], nbins, 0.0)
    np.testing.assert_array_equal(co[idx], cnt_o)
    nz = cnt_o > 0
    assert np.all(np.abs(fo[idx][nz].astype(np.float64) - mean_o[nz]) <= MEAN_RTOL * np.abs(mean_o[nz]))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_fold_below_256_bins_with_a_flux_that_is_no_number(ctx, bad):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(2)
    f = (1.0 + rng.normal(0.0, 3e-4, 3000)).astype(np.float32)
    f[1234] = bad
    args = [_dev(ctx, x) for x in (np.arange(3000) * CADENCE, f, rng.uniform(0.2, 1.0, 40))]
    folded, counts = g.gpfc_fold(ctx, *args, 100, 0.0)
    ctx.set_fold_config(layout=1)
    try:
        folded_e, counts_e = g.gpfc_fold(ctx, *args, 100, 0.0)
    finally:
        ctx.reset_fold_config()
    ctx.sync()
    assert torch.equal(counts, counts_e)
    assert torch.equal(torch.isfinite(folded), torch.isfinite(folded_e))


# profiles on which many starts and boxes lie near the top (ties, plateaus, slow ramps), and the ends
# of the width ranges and of the eight starts a lane takes
@pytest.mark.parametrize("nbins,w_min,w_max", [(256, 1, 1), (256, 2, 7), (256, 1, 8), (256, 9, 255), (300, 1, 100),
                                               (257, 3, 40), (40, 1, 40), (31, 1, 9)])
def test_box_scorer_on_ties_and_plateaus(ctx, nbins, w_min, w_max):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(nbins + w_max)
    i = np.arange(nbins)
    rows = [np.ones(nbins), 1.0 - 1e-3 * (i % 16 < 4), 1.0 - 1e-3 * (i < nbins // 2), 1.0 + 1e-5 * i,
            1.0 - 1e-3 * np.exp(-((i - 9.0) / 40.0) ** 2), 1.0 - 1e-3 * np.cos(2 * np.pi * i / nbins),
            1.0 - 1e-3 * (i == nbins - 1), 1.0 - 1e-3 * ((i < 2) | (i >= nbins - 3)),
            1.0 + 1e-7 * (i % 2), np.where(i % 3, 1.0, np.nan)]
    prof = np.array(rows * 5, np.float32)
    prof[10:20] += rng.normal(0, 1e-6, (10, nbins)).astype(np.float32)
    prof[20:30] += rng.normal(0, 1e-3, (10, nbins)).astype(np.float32)
    counts = np.full(prof.shape, 7, np.int32)
    counts[30:] = rng.integers(0, 500, (20, nbins))
    counts[np.isnan(prof)] = 0
    prof = np.where(counts > 0, prof, np.nan).astype(np.float32)
    sc, bs, bw = g.gpfc_score_box(ctx, _dev(ctx, prof), _dev(ctx, counts), w_min, w_max, 1e-4)
    ctx.sync()
    sc, bs, bw = (x.cpu().numpy() for x in (sc, bs, bw))
    sc_o, _, _ = oracle.box_snr_from_means(prof, counts, w_min, w_max, 1e-4)
    fin = np.isfinite(sc_o)
    np.testing.assert_array_equal(np.isfinite(sc), fin)
    # the general score: x = mean - reference in FP32 leaves 2^-24 of the level 1, 6e-8, in a bin's mean;
    # in units of sigma = 1e-4 and sqrt(counts of at most half the samples)
    n_tot = counts.sum(1).astype(np.float64)
    atol = 2.0 ** -24 / 1e-4 * np.sqrt(n_tot / 4.0)
    err = np.abs(sc[fin].astype(np.float64) - sc_o[fin])
    assert np.all(err <= BOX_RTOL * np.maximum(np.abs(sc_o[fin]), 1.0) + atol[fin])
    sums = np.where(counts > 0, prof.astype(np.float64) * counts, 0.0)
    for k in np.flatnonzero(fin):
        assert w_min <= bw[k] <= w_max and 0 <= bs[k] < nbins
        v = oracle.box_snr_at(sums[k], counts[k], int(bs[k]), int(bw[k]), 1e-4)
        assert abs(v - sc_o[k]) <= BOX_RTOL * max(abs(sc_o[k]), 1.0) + atol[k]


@pytest.mark.parametrize("n", [16383, 16384, 16385, 50001, 250001])
def test_decision_by_a_cluster_equals_one_block(ctx, n):
    """One star (a cluster of blocks from 16,384 periods) against the same star 20 times in a batch (a
    block each): whole numbers equal, sums within FP64 rounding."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(n)
    s = rng.normal(0, 1, n).astype(np.float32)
    for c in (0, n // 16 - 2, n // 3, n // 2 + 5, n - 6):
        s[c:c + 6] += 9.0
    s[77] = np.nan
    p = np.linspace(0.2, 30.0, n)
    one = g.peaks_to_numpy(*g.gpfc_peaks(ctx, _dev(ctx, s), _dev(ctx, p), max_peaks=16), 16)
    off = _dev(ctx, (np.arange(21) * n).astype(np.int64))
    many = g.peaks_to_numpy(*g.gpfc_peaks(ctx, _dev(ctx, np.tile(s, 20)), _dev(ctx, np.tile(p, 20)), off,
                                          max_peaks=16), 16)
    ctx.sync()
    a = one[0][0]
    for b, pk in ((many[0][0], many[1][0]), (many[0][19], many[1][19])):
        for key in ("best_index", "n_peaks", "n_listed", "truncated"):
            assert a[key] == b[key], key
        for key in ("sde", "mean", "sd"):
            assert abs(a[key] - b[key]) <= 1e-9 * max(1.0, abs(b[key])), key
        for key in ("index", "width", "harmonic", "height"):
            np.testing.assert_array_equal(one[1][0][key][:a["n_listed"]], pk[key][:a["n_listed"]])


@pytest.mark.parametrize("n_cad,nbins", [(1, 256), (127, 100), (6000, 256), (5003, 37)])
def test_generated_profiles_do_not_depend_on_the_batch(ctx, n_cad, nbins):
    """Few curves take 1,024 threads each, many take 256: the sums are integers, so equal."""
    import paper_2312_02063_gb300 as g
    sp = dict(lcsynth.TRAINING_SET, n_cadences=n_cad)
    many = g.gpfc_synth_profiles(ctx, 9, 40, 640, nbins, sp, want_period=True, want_std=True)
    for j in (0, 1, 2, 3, 639):
        one = g.gpfc_synth_profiles(ctx, 9, 40 + j, 1, nbins, sp, want_period=True, want_std=True)
        ctx.sync()
        for a, b in zip(one[:4], many[:4]):  # profile, counts, label, period
            assert torch.equal(torch.nan_to_num(a[0], 7.0), torch.nan_to_num(b[j], 7.0))


@pytest.mark.parametrize("lengths", [(2, 3, 4, 5, 7, 9, 12), (40, 41, 11, 300, 6), (1999, 2, 2001, 13, 64),
                                     (5000,)])
def test_detrending_of_short_and_odd_segments(ctx, lengths):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(len(lengths))
    t = np.concatenate([3.0 * k + sum(lengths[:k]) * CADENCE + np.arange(m) * CADENCE
                        for k, m in enumerate(lengths)])
    f = (1.0 + 1e-3 * np.sin(t) + rng.normal(0, 2e-4, len(t))).astype(np.float32)
    for edge in (0, 3):
        to, fo, so = g.gpfc_detrend(ctx, _dev(ctx, t), _dev(ctx, f), None, edge=edge)
        ctx.sync()
        r = oracle.detrend(t, f, None, edge=edge)
        np.testing.assert_array_equal(to.cpu().numpy(), r["times"])
        np.testing.assert_array_equal(so.cpu().numpy(), r["segment"])
        if len(r["times"]):
            err = np.abs(fo.cpu().numpy().astype(np.float64) - r["flux"]) / np.abs(r["flux"])
            assert err.max() <= FLUX_RTOL


@pytest.mark.parametrize("batch", [2, 130, 609, 2561])
def test_gradients_of_a_batch_are_the_sum_of_its_halves(ctx, batch):
    """The GEMMs of a large batch are not split over K, those of a small one are, into other pieces:
    the gradients of the whole batch against its halves' sum. FP32 sums in another order, and a rare
    BF16 rounding of a gradient that this moves across a tie: 1e-4 of a tensor's norm."""
    import paper_2312_02063_gb300 as g
    prof, lab = lcsynth.profiles_mixed(batch, seed=3)
    wd = {k: _dev(ctx, v) for k, v in lcsynth.cnn_init(3, bias_scale=0.05).items()}
    f = _dev(ctx, prof)
    logit, saved = g.gpfc_cnn_forward_train(ctx, f, wd)
    _, dl = g.gpfc_bce_with_logits(ctx, logit, _dev(ctx, lab.astype(np.float32)))
    whole = g.gpfc_cnn_backward(ctx, dl, wd, saved)
    h = batch // 2
    parts = []
    for a, b in ((0, h), (h, batch)):
        _, sv = g.gpfc_cnn_forward_train(ctx, f[a:b].contiguous(), wd)
        parts.append(g.gpfc_cnn_backward(ctx, dl[a:b].contiguous(), wd, sv))
    ctx.sync()
    for n in g.CNN_PARAM_NAMES:
        w, s = whole[n].double(), parts[0][n].double() + parts[1][n].double()
        assert float((w - s).norm()) <= 1e-4 * float(s.norm()) + 1e-12, n


# two rows of 32-bit words up to 65,536 samples, 64-bit words above; final bins about the 31 that a warp
# finishes at a time
@pytest.mark.parametrize("n,kind,nbins,merged", [
    (16383, "regular", 2048, 30), (16384, "regular", 1025, 31), (16385, "gaps", 3000, 32), (40000, "equal", 4096, 61),
    (65536, "regular", 4096, 62), (65537, "gaps", 4096, 63), (9000, "gaps", 1030, 2)])
def test_fine_bins_and_their_merging(ctx, n, kind, nbins, merged):
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(n)
    t = np.arange(n) * CADENCE + (3.3 * (np.arange(n) // 911) if kind == "gaps" else 0.0)
    if kind == "equal":
        t = np.full(n, 7.25)
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    p = np.r_[10 * CADENCE, rng.uniform(0.2, 1.0, 6), 17 * CADENCE]
    args = [_dev(ctx, x) for x in (t, f, p)]
    folded, counts = g.gpfc_fold(ctx, *args, nbins, 0.0)
    eq = g.gpfc_fold_equal_count(ctx, *args, merged, nbins, 0.0)
    ctx.sync()
    mean_o, cnt_o, _ = oracle.fold(t, f, p, nbins, 0.0)
    fo, co = folded.cpu().numpy().astype(np.float64), counts.cpu().numpy()
    np.testing.assert_array_equal(co, cnt_o)
    nz = cnt_o > 0
    assert np.all(np.abs(fo[nz] - mean_o[nz]) <= MEAN_RTOL * np.abs(mean_o[nz]))
    eq_o, _ = oracle.fold_equal_count(t, f, p, nbins, merged, 0.0)
    assert np.all(np.abs(eq.cpu().numpy() - eq_o) <= MEAN_RTOL * np.abs(eq_o))
