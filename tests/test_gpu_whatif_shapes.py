"""What-if over the block shapes of the pair kernel (few and many candidates and pending requests)
and both candidate passes, and admission with budgets, totals and objectives that are NaN, infinite,
zero of either sign or exactly met: the mask equals the fp64 predicate on the device's own T_new and
shares, and T_new and shares agree with the oracle within 1e-12."""

import numpy as np
import pytest

import oracle
import test_gpu_attribute as base

pytestmark = pytest.mark.gpu

lv = base.lv
ctx = base.ctx


def _pending(rng, n):
    ph = (rng.random(n) < 0.3).astype(np.int32)
    p = np.where(ph == 1, rng.integers(1, 5000, n), 1).astype(np.int32)
    c = np.where(ph == 1, 0, rng.integers(0, 50000, n)).astype(np.int32)
    return p, c, ph


def _whatif(lv, ctx, w, p, c, ph, adm=None):
    import torch
    d = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    shape = (len(p), w.n_batch)
    T, S = (torch.full(shape, float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
    b, model = base._dev(lv, w, tenant=False), lv.make_model(w.coef, w.split)
    A = None
    if adm is None:
        lv.lv_whatif(ctx, model, b, d(p), d(c), d(ph), T, S)
    else:
        ten, L, B, slo = adm
        A = torch.full(shape, 7, dtype=torch.uint8, device="cuda")
        lv.lv_whatif_admit(ctx, model, b, d(p), d(c), d(ph), d(ten), d(L), d(B), slo, A, T, S)
        A = A.cpu().numpy()
    assert ctx.status() == lv.LV_OK
    return T.cpu().numpy(), S.cpu().numpy(), A


@pytest.mark.parametrize("nc,npend", [(1, 1), (5, 700), (31, 33), (33, 5), (65, 130), (129, 40), (2433, 3), (9728, 2), (9729, 3),
                                     (300, 1000)])
def test_shapes(lv, ctx, nc, npend):
    rng = np.random.default_rng(nc * 1000 + npend)
    sizes = rng.integers(0, 300, nc)
    sizes[0] = 700
    w = base._from_sizes(rng, sizes, pre=0.05)
    p, c, ph = _pending(rng, npend)
    T, S, _ = _whatif(lv, ctx, w, p, c, ph)
    T_o, S_o = oracle.whatif(w.offsets, w.p, w.c, w.phase, p, c, ph, w.split, w.coef)
    assert np.max(np.abs(T - T_o) / T_o) <= 1e-12 and np.max(np.abs(S - S_o) / S_o) <= 1e-12


@pytest.mark.parametrize("sizes", [[4097, 0, 4096, 4099], [1, 1023, 1024, 1025, 1026, 2047, 2049], [8191, 8192, 8193, 8195],
                                   [300_001], [3, 5, 100_002], [4096] * 305])
def test_large_candidates(lv, ctx, sizes):
    """Candidates of one and of several turns of a block's loads, in blocks of 128 and of 512 threads, and arrays that
    end inside a quad."""
    rng = np.random.default_rng(len(sizes))
    w = base._from_sizes(rng, np.array(sizes), pre=0.02)
    p, c, ph = _pending(rng, 40)
    T, S, _ = _whatif(lv, ctx, w, p, c, ph)
    T_o, S_o = oracle.whatif(w.offsets, w.p, w.c, w.phase, p, c, ph, w.split, w.coef)
    assert np.max(np.abs(T - T_o) / T_o) <= 1e-12 and np.max(np.abs(S - S_o) / S_o) <= 1e-12


@pytest.mark.parametrize("split", [-2 ** 63, -2 ** 63 + 1, -1, 0, 1, 2 ** 31, 2 ** 63 - 1])
def test_extreme_splits(lv, ctx, split):
    """Splits that every batch or none meets: the regime is S1 + p >= split in 64 bits."""
    rng = np.random.default_rng(43)
    w = base._from_sizes(rng, rng.integers(0, 60, 70), pre=0.05)
    w.split[:] = split
    p, c, ph = _pending(rng, 90)
    T, S, _ = _whatif(lv, ctx, w, p, c, ph)
    T_o, S_o = oracle.whatif(w.offsets, w.p, w.c, w.phase, p, c, ph, w.split, w.coef)
    assert np.max(np.abs(T - T_o) / T_o) <= 1e-12 and np.max(np.abs(S - S_o) / S_o) <= 1e-12


@pytest.mark.parametrize("slo", [0.004, 0.0, -0.0, float("nan"), float("inf"), float("-inf")])
def test_admission_edges(lv, ctx, slo):
    rng = np.random.default_rng(41)
    w = base._from_sizes(rng, rng.integers(1, 60, 70), pre=0.02)
    p, c, ph = _pending(rng, 90)
    inf, nan = float("inf"), float("nan")
    neg_nan, full_nan = np.array([0xfff8000000000000, 0xffffffffffffffff], np.uint64).view(np.float64)
    L = np.array([0.0, -0.0, 1e-3, nan, inf, -inf, 5.0, 0.0, 1e-3, neg_nan, full_nan, neg_nan, 0.0])
    B = np.array([0.0, -0.0, 2e-3, 1.0, inf, inf, nan, 1e-3, -inf, 1.0, inf, full_nan, full_nan])
    ten = rng.integers(0, len(L), len(p)).astype(np.int32)
    T, S, _ = _whatif(lv, ctx, w, p, c, ph)
    B[7], L[7] = S[ten == 7][0, 3], 0.0   # a budget met exactly
    T, S, A = _whatif(lv, ctx, w, p, c, ph, (ten, L, B, slo))
    with np.errstate(invalid="ignore"):
        want = (L[ten][:, None] + S <= B[ten][:, None]) & (T <= slo)
    assert np.array_equal(A, want.astype(np.uint8))
    if slo == inf:
        assert A[ten == 7][0, 3] == 1
