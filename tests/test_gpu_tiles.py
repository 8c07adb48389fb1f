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


@pytest.mark.parametrize("p_max", [1, 8192, 8193, 1 << 23])
@pytest.mark.parametrize("share", [1e-3, 1.0])
@pytest.mark.parametrize("lo,hi,n", [(0, 9, 9000), (1, 300, 900), (900, 1530, 60)])
def test_long_contexts(lv, ctx, p_max, share, lo, hi, n):
    """Contexts of 2^23 tokens and more, up to the type's largest, in some tiles and in all, beside prefills of
    several lengths."""
    import torch
    rng = np.random.default_rng(p_max + hi)
    w = base._from_sizes(rng, rng.integers(lo, hi + 1, n), nt=20, pre=0.3)
    at = rng.random(w.n_req) < share
    w.c[at] = rng.integers(1 << 23, 1 << 31, int(at.sum()))
    w.c[rng.integers(0, w.n_req, 50)] = (1 << 31) - 1
    w.p[w.phase == 1] = np.where(rng.random(int((w.phase == 1).sum())) < 0.9, p_max, 2)
    _check(lv, ctx, w)
    b = base._dev(lv, w, tenant=False)
    bf = torch.empty((5, w.n_batch), dtype=torch.int64, device="cuda")
    lv.lv_features(ctx, b, model=lv.make_model(w.coef, w.split), batch_feat=bf)
    assert ctx.status() == lv.LV_OK
    assert np.array_equal(bf.cpu().numpy(), oracle.batch_features(w.offsets, w.p, w.c, w.phase, w.split)[0])


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


def _queued(kind):
    """Sizes of an input of more than one tile per warp (3.8e6 positions) with batches that no tile holds."""
    rng = np.random.default_rng(50)
    small = rng.integers(0, 9, 460_000)
    edges = np.array([1533, 1536, 1537, 1540, 4095, 4096, 4097, 24_575, 24_576, 24_577, 100_001])
    if kind == "few":
        s = np.concatenate([small, edges, rng.integers(1500, 70_000, 20)])
    elif kind == "warps":
        s = rng.integers(1537, 1800, 4_700)     # enough for every warp of the chip
    elif kind == "teams":
        s = np.concatenate([rng.integers(1537, 4000, 900), rng.integers(4097, 9000, 500)])  # enough for teams
    elif kind == "ctas":
        s = rng.integers(24_577, 28_000, 200)
    else:
        s = np.concatenate([small[:1000], edges, rng.integers(1537, 1600, 4_600), rng.integers(4097, 9000, 400),
                            rng.integers(24_577, 28_000, 160)])
    rng.shuffle(s)
    return s


_MODES = ["f64", "f64_unaligned", "fp64_arith", "f32", "f32_unaligned"]


def _check_mode(lv, ctx, w, mode):
    """Two calls, alike bit for bit, against the oracle.  fp32: within 1e-5, the stated bound."""
    import torch
    b, model = base._dev(lv, w), lv.make_model(w.coef, w.split)
    f32, at = mode.startswith("f32"), 1 if "unaligned" in mode else 0
    dt = torch.float32 if f32 else torch.float64
    outs = []
    for _ in range(2):
        T = torch.full((w.n_batch + at,), float("nan"), dtype=dt, device="cuda")[at:]
        S = torch.full((w.n_req + at,), float("nan"), dtype=dt, device="cuda")[at:]
        acc = lv.TenantAcc(ctx, w.n_tenants)
        ctx.set_arith(1 if mode == "fp64_arith" else 0)
        (lv.lv_attribute_f32 if f32 else lv.lv_attribute)(ctx, model, b, T, S, acc)
        L = torch.empty(w.n_tenants, dtype=torch.float64, device="cuda")
        lv.lv_tenant_totals(ctx, acc, L)
        assert ctx.status() == lv.LV_OK
        ctx.set_arith(0)
        outs.append([x.cpu().numpy().astype(np.float64) for x in (T, S, L)])
    for x, y in zip(*outs):
        assert np.array_equal(x, y)
    T, S, L = outs[0]
    if not f32:
        base._check_parity(w, T, S, L)
        return
    T_o, s_o = oracle.attribute(w.offsets, w.p, w.c, w.phase, w.split, w.coef)
    nz = T_o != 0
    assert np.all(T[~nz] == 0) and np.max(np.abs(T[nz] - T_o[nz]) / T_o[nz]) <= 1e-5
    assert np.max(np.abs(S - s_o) / s_o) <= 1e-5
    L_o = oracle.tenant_totals(s_o, w.tenant, w.n_tenants)
    assert np.max(np.abs(L - L_o) / L_o) <= 1e-5


@pytest.mark.parametrize("kind", ["few", "warps", "teams", "ctas", "all"])
@pytest.mark.parametrize("mode", _MODES)
def test_queued_batches(lv, ctx, kind, mode):
    """Batches that no tile holds, by warps, teams and whole CTAs.  Each call twice: the queue of the second starts
    where the first left it."""
    rng = np.random.default_rng(51)
    _check_mode(lv, ctx, base._from_sizes(rng, _queued(kind), nt=600, pre=0.02), mode)


@pytest.mark.parametrize("lo,hi,n", [(0, 2, 9000), (1, 8, 6000), (30, 50, 900), (1240, 1256, 200), (1528, 1544, 150),
                                     (513, 5000, 200)])
@pytest.mark.parametrize("mode", _MODES[1:])
def test_modes_around_the_tile(lv, ctx, lo, hi, n, mode):
    rng = np.random.default_rng(hi)
    _check_mode(lv, ctx, base._from_sizes(rng, rng.integers(lo, hi + 1, n), nt=9, pre=0.1), mode)


@pytest.mark.parametrize("kind", ["few", "warps", "teams", "ctas", "all"])
def test_queued_batches_features_and_noalloc(lv, ctx, kind):
    """The same inputs' batch features, and lv_attribute_noalloc's T and shares bit for bit those of lv_attribute."""
    import ctypes
    import torch
    w = base._from_sizes(np.random.default_rng(52), np.concatenate([_queued(kind)] * 2), pre=0.02)
    b, model = base._dev(lv, w, tenant=False), lv.make_model(w.coef, w.split)
    bf = torch.empty((5, w.n_batch), dtype=torch.int64, device="cuda")
    bs = torch.empty(w.n_batch, dtype=torch.uint8, device="cuda")
    lv.lv_features(ctx, b, model=model, batch_feat=bf, batch_seg=bs)
    feat, seg = oracle.batch_features(w.offsets, w.p, w.c, w.phase, w.split)
    assert ctx.status() == lv.LV_OK
    assert np.array_equal(bf.cpu().numpy(), feat) and np.array_equal(bs.cpu().numpy(), seg)
    T, S = base._run(lv, ctx, w, acc=False)[:2]
    status = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    bst = b.struct()
    for _ in range(2):
        Tn = torch.full((w.n_batch,), float("nan"), dtype=torch.float64, device="cuda")
        Sn = torch.full((w.n_req,), float("nan"), dtype=torch.float64, device="cuda")
        rc = lv.lib().lv_attribute_noalloc(ctypes.byref(model), ctypes.byref(bst), Tn.data_ptr(), Sn.data_ptr(),
                                           status.data_ptr(), torch.cuda.current_stream().cuda_stream)
        assert rc == lv.LV_OK and int(status.item()) == 0
        assert np.array_equal(Tn.cpu().numpy(), T) and np.array_equal(Sn.cpu().numpy(), S)


@pytest.mark.parametrize("kind", ["few", "teams"])
def test_invalid_values_in_queued_batches(lv, ctx, kind):
    """Negative p and c count as 0, tenants out of range as the nearest; the call reports them."""
    rng = np.random.default_rng(53)
    w = base._from_sizes(rng, _queued(kind), nt=7, pre=0.02)
    big = np.flatnonzero(np.diff(w.offsets) > 1536)
    at = w.offsets[rng.choice(big, 30)] + rng.integers(0, 1537, 30)
    w.p[at[:10]], w.c[at[10:20]], w.tenant[at[20:25]], w.tenant[at[25:]] = -5, -(1 << 31), -1, 7
    T, S, L, st = base._run(lv, ctx, w)
    assert st == lv.LV_EDATA
    w.p[:], w.c[:], w.tenant[:] = np.maximum(w.p, 0), np.maximum(w.c, 0), np.clip(w.tenant, 0, 6)
    base._check_parity(w, T, S, L)
