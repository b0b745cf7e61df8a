"""The one-word fold (sum and count of a bin in one shared-memory word, checked segment by
segment) against the two-word reduction fold and the FP64 oracle: both sum the same fixed-point
flux exactly and round once, so every output must be bit-identical, whatever the segment, the
fallback to two passes and the block shape."""
import numpy as np
import pytest
import torch

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


def _times(kind, n, rng):
    t = np.arange(n) * CADENCE
    if kind == "gaps":
        t = t + 3.3 * (np.arange(n) // 911)
    elif kind == "unsorted":
        t = rng.uniform(0.0, 900.0, n)
    elif kind == "equal":  # every sample in one bin of every period: only two passes can fold it
        t = np.full(n, 7.25)
    elif kind == "nights":  # a third of each day, at 24 s
        t = np.arange(n) // 1200 + (np.arange(n) % 1200) * (1.0 / 3600.0)
    return t


def _both(ctx, t, f, p, nbins):
    import paper_2312_02063_gb300 as g
    args = [_dev(ctx, x) for x in (t, f, p)]
    out = []
    try:
        for two_words in (False, True):
            if two_words:
                ctx.set_fold_config(warps=1, layout=g.LAYOUT_RED32)
            folded, counts = g.gpfc_fold(ctx, *args, nbins, 0.0)
            ctx.sync()
            out.append((folded.cpu().numpy(), counts.cpu().numpy()))
    finally:
        ctx.reset_fold_config()
    return out


# lengths about the tile (2,048), the segment (16 tiles), the chunk (65,520) and the groups of 16;
# period counts about the group (32) and the block (192)
@pytest.mark.parametrize("n,kind,n_periods,nbins", [
    (1, "regular", 1, 256), (15, "regular", 33, 256), (17, "unsorted", 31, 256), (300, "gaps", 193, 256),
    (2047, "regular", 200, 256), (2049, "gaps", 64, 256), (4096, "equal", 40, 256), (6000, "unsorted", 700, 256),
    (32768, "regular", 33, 256), (32769, "gaps", 193, 256), (65519, "regular", 96, 256), (65521, "gaps", 96, 256),
    (70001, "unsorted", 65, 256), (140000, "nights", 40, 256), (5001, "regular", 129, 300), (40000, "gaps", 97, 512),
    (9000, "equal", 33, 512), (33000, "nights", 65, 1000), (20011, "unsorted", 34, 1024), (66000, "gaps", 33, 300)])
def test_equals_two_word_fold(ctx, n, kind, n_periods, nbins):
    rng = np.random.default_rng(n + nbins)
    t = _times(kind, n, rng)
    f = (1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32)
    p = rng.uniform(0.2, 1.0, n_periods)
    # multiples of the cadence: the samples pile up in 10, 17 and 49 bins
    for i, m in enumerate((10, 17, 49)):
        if i < n_periods:
            p[i] = m * CADENCE
    (fa, ca), (fb, cb) = _both(ctx, t, f, p, nbins)
    np.testing.assert_array_equal(ca, cb)
    np.testing.assert_array_equal(fa, fb)
    _, cnt, _ = oracle.fold(t, f, p[:5], nbins, 0.0)
    np.testing.assert_array_equal(ca[:5], cnt)


def test_batch_of_uneven_stars_equals_single_stars(ctx):
    """Stars of 1 to 70,000 samples and 1 to 900 periods in one batch: every score equals the star's
    own search, in the one-word and in the two-word fold."""
    import paper_2312_02063_gb300 as g
    rng = np.random.default_rng(8)
    ns, ps = [1, 40, 513, 2048, 5000, 33000, 70000], [1, 500, 193, 192, 900, 64, 300]
    ts = [_times("gaps", n, rng) for n in ns]
    fs = [(1.0 + rng.normal(0.0, 3e-4, n)).astype(np.float32) for n in ns]
    gs = [rng.uniform(0.2, 1.0, m) for m in ps]
    off = lambda xs: np.concatenate([[0], np.cumsum([len(x) for x in xs])]).astype(np.int64)  # noqa: E731
    d = [_dev(ctx, x) for x in (off(ts), np.concatenate(ts), np.concatenate(fs), off(gs), np.concatenate(gs),
                                np.zeros(len(ns)))]
    score, bi, _ = g.gpfc_search_batched(ctx, d[0], d[1], d[2], d[3], d[4], 256, d[5], g.SCORER_BOX, w_max=40)
    ctx.sync()
    score, o = score.cpu().numpy(), off(gs)
    for s in range(len(ns)):
        one, k, _ = g.gpfc_search(ctx, _dev(ctx, ts[s]), _dev(ctx, fs[s]), _dev(ctx, gs[s]), 256, 0.0, g.SCORER_BOX,
                                  w_max=40)
        try:
            ctx.set_fold_config(warps=1, layout=g.LAYOUT_RED32)
            two, _, _ = g.gpfc_search(ctx, _dev(ctx, ts[s]), _dev(ctx, fs[s]), _dev(ctx, gs[s]), 256, 0.0,
                                      g.SCORER_BOX, w_max=40)
        finally:
            ctx.reset_fold_config()
        ctx.sync()
        np.testing.assert_array_equal(score[o[s]:o[s + 1]], one.cpu().numpy())
        np.testing.assert_array_equal(one.cpu().numpy(), two.cpu().numpy())
        assert int(bi[s].item()) == int(k.item())
