"""The tile kernel at the edges of its tiles: batch sizes around a tile's staged requests and
the sizes that a warp or the whole CTA walks, request arrays that end inside a quad, values too
large for the 32-bit prefixes, and tenant contributions on both sides of the hot-table limits.

Tolerances as in test_gpu_attribute: 1e-12 relative against the oracle, tenant totals equal to
the correctly rounded exact sums of the shares.
"""

import numpy as np
import pytest

import oracle
import test_gpu_attribute as base

pytestmark = pytest.mark.gpu

lv = base.lv
ctx = base.ctx


def _check(lv, ctx, w, acc=True):
    T, share, L, st = base._run(lv, ctx, w, acc=acc)
    assert st == lv.LV_OK
    base._check_parity(w, T, share, L)


@pytest.mark.parametrize("lo,hi,n", [(0, 2, 6000), (1, 8, 3000), (30, 50, 900), (250, 262, 400), (284, 292, 300),
                                     (500, 520, 300), (1240, 1256, 200), (1528, 1544, 150), (513, 5000, 200)])
@pytest.mark.parametrize("cut", [0, 1, 3])
def test_sizes_around_the_tile(lv, ctx, lo, hi, n, cut):
    """Sizes lo..hi, the last batch cut so that the arrays end 0, 1 or 3 requests into a quad."""
    rng = np.random.default_rng(1000 * hi + cut)
    sizes = rng.integers(lo, hi + 1, n)
    sizes[-1] = 8
    sizes[-1] += (cut - int(sizes.sum())) % 4
    _check(lv, ctx, base._from_sizes(rng, sizes, nt=7, pre=0.1))


def test_more_large_batches_than_a_cta_keeps(lv, ctx):
    rng = np.random.default_rng(12)
    _check(lv, ctx, base._from_sizes(rng, rng.integers(1100, 1140, 11_000), nt=3, pre=0.02))


@pytest.mark.parametrize("field", ["p", "c"])
def test_values_beyond_the_prefix_words(lv, ctx, field):
    """One request of 2^23 or more per few hundred: its tile's batches are walked one by one."""
    rng = np.random.default_rng(13)
    w = base._from_sizes(rng, rng.integers(1, 40, 4000), nt=600, pre=0.1)
    at = rng.integers(0, w.n_req, 200)
    getattr(w, field)[at] = rng.integers(1 << 23, 1 << 24, 200)
    if field == "p":
        w.phase[at] = 1
    _check(lv, ctx, w)


@pytest.mark.parametrize("nt", [1, 511, 512, 513, 1536, 1537, 3000])
@pytest.mark.parametrize("scale", [1e-4, 1.0, 300.0])
def test_tenants_and_share_magnitudes(lv, ctx, nt, scale):
    """Shares below 2^-20 s (rounded to the 2^-72 s grid), common ones, and ones of 2^-9 s and
    more (more than two words), with hot tenants only and with cold ones."""
    rng = np.random.default_rng(14)
    w = base._from_sizes(rng, rng.integers(1, 200, 1500), nt=nt, pre=0.1)
    w.coef[:] *= scale
    _check(lv, ctx, w)


def test_features_match_attribution_sums(lv, ctx):
    import torch
    rng = np.random.default_rng(15)
    w = base._from_sizes(rng, rng.integers(0, 1100, 500), pre=0.1)
    w.c[::997] = 1 << 30
    b = base._dev(lv, w, tenant=False)
    bf = torch.empty((5, w.n_batch), dtype=torch.int64, device="cuda")
    bs = torch.empty(w.n_batch, dtype=torch.uint8, device="cuda")
    lv.lv_features(ctx, b, model=lv.make_model(w.coef, w.split), batch_feat=bf, batch_seg=bs)
    assert ctx.status() == lv.LV_OK
    feat, seg = oracle.batch_features(w.offsets, w.p, w.c, w.phase, w.split)
    assert np.array_equal(bf.cpu().numpy(), feat) and np.array_equal(bs.cpu().numpy(), seg)


@pytest.mark.parametrize("lo,hi,n,cut", [(0, 1, 1_200_001, 1), (1, 40, 300_002, 0), (2470, 2500, 4003, 3),
                                         (2548, 2566, 3500, 1), (3000, 6000, 60, 0)])
def test_feature_sizes_around_the_tile(lv, ctx, lo, hi, n, cut):
    """The feature pass has tiles of its own: exact sums at the edges of their positions and
    requests (inputs of more than 7.6e6 positions, so that the tiles have their full size)."""
    import torch
    rng = np.random.default_rng(100 * hi + cut)
    sizes = rng.integers(lo, hi + 1, n)
    sizes[-1] = 8
    sizes[-1] += (cut - int(sizes.sum())) % 4
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    m = int(off[-1])
    ph = (rng.random(m) < 0.002).astype(np.int32)
    p, c = np.where(ph == 1, rng.integers(1, 8192, m), 1).astype(np.int32), rng.integers(0, 1 << 17, m).astype(np.int32)
    coef = np.ones((2, 2, 5))
    model = lv.make_model(coef, (256, 300))
    feat = torch.full((5, n), -1, dtype=torch.int64, device="cuda")
    seg = torch.full((n,), 9, dtype=torch.uint8, device="cuda")
    lv.lv_features(ctx, lv.batches_to_device(p, c, ph, off), model=model, batch_feat=feat, batch_seg=seg)
    assert ctx.status() == lv.LV_OK
    want, want_seg = oracle.batch_features(off, p, c, ph, (256, 300))
    assert np.array_equal(feat.cpu().numpy(), want) and np.array_equal(seg.cpu().numpy(), want_seg)


@pytest.mark.parametrize("at", [0, 1, 2, 499_996, 499_997, 499_998, 499_999, 1_000_001, 1_000_002])
def test_offsets_out_of_order_are_seen(lv, ctx, at):
    """One offset below the one before it, in each place of a thread's four and in the last ones (an input
    whose tile bounds have a kernel of their own)."""
    import torch
    n = 1_000_002
    off = np.arange(n + 1, dtype=np.int64)
    one, zero = np.ones(n, np.int32), np.zeros(n, np.int32)
    feat = torch.zeros((5, n), dtype=torch.int64, device="cuda")
    seg = torch.zeros(n, dtype=torch.uint8, device="cuda")
    model = lv.make_model(np.ones((2, 2, 5)), (256, 300))
    for bad in (off[at] - 2, None):
        o = off.copy()
        o[at] = off[at] if bad is None else bad
        lv.lv_features(ctx, lv.batches_to_device(one, zero, zero, o), model=model, batch_feat=feat, batch_seg=seg)
        assert ctx.status() == (lv.LV_OK if bad is None else lv.LV_EDATA)
