"""Edges of the accuracy metrics: the digits of the exact division at the ends
of the divisor's and the difference's ranges, and batch counts on either
side of a doubling of the select's buckets.  Percentiles exact, R^2 and the mean
relative error within 1e-12, as for every other input."""

import numpy as np
import pytest

import oracle
from test_gpu_accuracy import _check_accuracy, _dev, ctx, lv  # noqa: F401

pytestmark = pytest.mark.gpu

_TOP = 2 ** 52
_EDGES = [0, 1, 2, (1 << 29) - 1, 1 << 29, (1 << 29) + 1, (1 << 51) - 1, 1 << 51, _TOP - (1 << 29) - 1,
          _TOP - (1 << 29), _TOP - 2, _TOP - 1]


def test_division_digit_edges(lv, ctx):  # noqa: F811
    """rel = (T - y) / y with T = y + d exact, y and d at mantissas next to
    a power of two, to a carry of the truncated divisor and to their middles."""
    for my in _EDGES:
        y = (_TOP + my) / _TOP
        for md in _EDGES:
            for T in (y + (_TOP + md) / _TOP * 0.25, y - (_TOP + md) / _TOP * 0.25):
                g = lv.lv_accuracy(ctx, _dev([y]), _dev([T]))
                assert g["p50"] == g["p99"] == abs(T - y) / y, (my, md, T)


@pytest.mark.parametrize("n", [(1 << 21) - 1, 1 << 21, (1 << 21) + 1, 4_300_007])
def test_bucket_sizes(lv, ctx, n):  # noqa: F811
    """Lognormal errors: the busiest second-digit bins of these counts hold
    around 64 samples and more, below and above the buckets' size."""
    rng = np.random.default_rng(n)
    T = rng.lognormal(-3.0, 0.6, n)
    y = T * rng.lognormal(0.0, 0.1, n)
    _check_accuracy(lv.lv_accuracy(ctx, _dev(y), _dev(T)), oracle.accuracy(y, T))


@pytest.mark.parametrize("n,k", [(1, 1), (50, 1), (50, 30), (20_000, 7), (20_000, 500), (300_000, 100_000)])
@pytest.mark.parametrize("T_inf", [False, True])
def test_infinite_latencies(lv, ctx, n, k, T_inf):  # noqa: F811
    """y = +inf counts as a sample; its relative error is a NaN (inf / inf, or inf - inf), which ranks above
    every number, whatever sign the arithmetic gives it."""
    rng = np.random.default_rng(n + k)
    T = rng.lognormal(-3.0, 0.6, n)
    y = T * rng.lognormal(0.0, 0.1, n)
    at = rng.choice(n, k, replace=False)
    y[at] = np.inf
    if T_inf:
        T[at[::2]] = np.inf
    g = lv.lv_accuracy(ctx, _dev(y), _dev(T))
    with np.errstate(invalid="ignore"):
        rel = np.sort(np.abs(T - y) / y)  # NaN last
    assert g["n"] == n and np.isnan(g["mean_rel"]) and np.isnan(g["r2_ssr"]) and np.isnan(g["r2_corr"])
    for name, q in (("p50", 50), ("p90", 90), ("p99", 99)):
        want = rel[-(-q * n // 100) - 1]
        assert g[name] == want or (np.isnan(g[name]) and np.isnan(want)), name
