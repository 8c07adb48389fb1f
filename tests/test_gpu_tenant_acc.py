"""lv_tenant_accumulate at the edges of its kernel: sizes around a thread's four shares and a CTA's
turn, tenant counts on both sides of the hot-table limits, and shares of every kind (zero, subnormal,
negative, below the 2^-72 s grid, 2^-9 s and more).  Totals equal the exact sums bit for bit."""

import numpy as np
import pytest

import test_gpu_attribute as base

pytestmark = pytest.mark.gpu

lv = base.lv
ctx = base.ctx


def _totals(lv, ctx, share, ten, nt):
    import torch
    acc = lv.TenantAcc(ctx, nt)
    lv.lv_tenant_accumulate(ctx, acc, torch.as_tensor(share, device="cuda"), torch.as_tensor(ten, device="cuda"))
    L = torch.empty(nt, dtype=torch.float64, device="cuda")
    lv.lv_tenant_totals(ctx, acc, L)
    assert ctx.status() == lv.LV_OK
    return L.cpu().numpy()


@pytest.mark.parametrize("n,nt", [(1, 1), (1023, 511), (1025, 512), (4096, 513), (4097, 16), (70_000, 273),
                                  (200_000, 600), (200_000, 800), (2_200_000, 8192), (2_200_000, 8193)])
def test_exact_totals(lv, ctx, n, nt):
    rng = np.random.default_rng(n + nt)
    share = np.exp(rng.normal(-11.0, 2.0, n))
    k = min(n, 64)
    odd = np.array([0.0, -0.0, 5e-324, -3e-310, 2.0 ** -73, 3.0 * 2.0 ** -74, -(2.0 ** -72), 2.0 ** -9, -1.5e-3, 0.75,
                    1e6, -1e6, 2.0 ** -20, np.nextafter(2.0 ** -9, 0)])
    share[rng.choice(n, k, replace=False)] = odd[rng.integers(0, len(odd), k)]
    ten = np.minimum(rng.integers(0, nt, n), rng.integers(0, nt, n)).astype(np.int32)
    L = _totals(lv, ctx, share, ten, nt)
    order = np.argsort(ten, kind="stable")
    bounds = np.searchsorted(ten[order], np.arange(nt + 1))
    for u in np.unique(np.concatenate([np.arange(min(nt, 20)), np.arange(max(nt - 20, 0), nt), [min(511, nt - 1)]])):
        if bounds[u + 1] - bounds[u] < 200_000:
            assert L[u] == base.exact_tenant_total(share[order[bounds[u]:bounds[u + 1]]]), u
