"""The calls that may be captured into a CUDA graph, at sizes with kernels launched before the one ahead
has ended (tile bounds, tiles, the queue of large batches, tenant totals; what-if candidates and pairs):
captured once, each of several replays in a row gives the eager call's outputs bit for bit."""

import numpy as np
import pytest

import test_gpu_attribute as base

pytestmark = pytest.mark.gpu

lv = base.lv
ctx = base.ctx


def _replay(call, outs, ctx, lv):
    """call(stream) once eagerly and three times from a graph, from outputs wiped before; the outputs must agree."""
    import torch
    call(None)
    torch.cuda.synchronize()
    want = [x.clone() for x in outs]
    cs = torch.cuda.Stream()
    cs.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(cs):
        call(cs)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=cs):
        call(cs)
    for _ in range(3):
        for x in outs:
            x.fill_(7)
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        for x, w in zip(outs, want):
            assert torch.equal(x.view(torch.uint8), w.view(torch.uint8))
    assert ctx.status() == lv.LV_OK
    call(None)  # and an eager call after the replays
    torch.cuda.synchronize()
    for x, w in zip(outs, want):
        assert torch.equal(x.view(torch.uint8), w.view(torch.uint8))


def _sizes(kind):
    rng = np.random.default_rng(60)
    if kind == "search":
        return rng.integers(0, 60, 20_000)
    s = rng.integers(0, 9, 460_000)
    if kind == "queue":
        s[rng.choice(len(s), 40, replace=False)] = rng.integers(1537, 70_000, 40)
    return s


@pytest.mark.parametrize("kind", ["search", "tiles", "queue"])
@pytest.mark.parametrize("nt", [16, 3000])
@pytest.mark.parametrize("f32", [False, True])
def test_attribution_and_totals(lv, ctx, kind, nt, f32):
    import torch
    w = base._from_sizes(np.random.default_rng(61), _sizes(kind), nt=nt, pre=0.02)
    b, model = base._dev(lv, w), lv.make_model(w.coef, w.split)
    dt = torch.float32 if f32 else torch.float64
    T, S = torch.empty(w.n_batch, dtype=dt, device="cuda"), torch.empty(w.n_req, dtype=dt, device="cuda")
    L, acc = torch.empty(nt, dtype=torch.float64, device="cuda"), lv.TenantAcc(ctx, nt)

    def call(stream):
        acc.reset(stream)
        (lv.lv_attribute_f32 if f32 else lv.lv_attribute)(ctx, model, b, T, S, acc, stream=stream)
        lv.lv_tenant_totals(ctx, acc, L, stream=stream)

    _replay(call, [T, S, L], ctx, lv)


@pytest.mark.parametrize("kind", ["search", "queue"])
def test_features_and_latency(lv, ctx, kind):
    import torch
    w = base._from_sizes(np.random.default_rng(62), np.concatenate([_sizes(kind)] * 3), pre=0.02)
    b, model = base._dev(lv, w, tenant=False), lv.make_model(w.coef, w.split)
    rf = torch.empty((3, w.n_req), dtype=torch.int64, device="cuda")
    bf = torch.empty((5, w.n_batch), dtype=torch.int64, device="cuda")
    bs = torch.empty(w.n_batch, dtype=torch.uint8, device="cuda")
    T = torch.empty(w.n_batch, dtype=torch.float64, device="cuda")

    def call(stream):
        lv.lv_features(ctx, b, arch=w.arch, model=model, req_feat=rf, batch_feat=bf, batch_seg=bs, stream=stream)
        lv.lv_batch_latency(ctx, model, bf, bs, T, stream=stream)

    _replay(call, [rf, bf, bs, T], ctx, lv)


@pytest.mark.parametrize("nt", [16, 3000])
def test_accumulate(lv, ctx, nt):
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(63)
    share = torch.rand(1_000_003, generator=g, device="cuda", dtype=torch.float64) * 1e-3
    ten = torch.randint(0, nt, (1_000_003,), generator=g, device="cuda", dtype=torch.int32)
    L, acc = torch.empty(nt, dtype=torch.float64, device="cuda"), lv.TenantAcc(ctx, nt)

    def call(stream):
        acc.reset(stream)
        lv.lv_tenant_accumulate(ctx, acc, share, ten, stream=stream)
        lv.lv_tenant_totals(ctx, acc, L, stream=stream)

    _replay(call, [L], ctx, lv)


@pytest.mark.parametrize("nc,npend", [(24, 500), (1024, 300), (10_000, 40)])
@pytest.mark.parametrize("admit", [False, True])
def test_whatif(lv, ctx, nc, npend, admit):
    """Candidates by a block each and, for 10,000, by the tile pass."""
    import torch
    rng = np.random.default_rng(64)
    w = base._from_sizes(rng, rng.integers(0, 200, nc), pre=0.02)
    b, model = base._dev(lv, w, tenant=False), lv.make_model(w.coef, w.split)
    d = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    ph = (rng.random(npend) < 0.3).astype(np.int32)
    p, c = d(np.where(ph == 1, rng.integers(1, 5000, npend), 1).astype(np.int32)), d(rng.integers(0, 50000, npend, np.int32))
    ten, L, B = d(rng.integers(0, 8, npend, np.int32)), d(rng.random(8) * 1e-3), d(rng.random(8) * 1e-2)
    T, S = (torch.empty((npend, nc), dtype=torch.float64, device="cuda") for _ in range(2))
    A = torch.empty((npend, nc), dtype=torch.uint8, device="cuda")

    def call(stream):
        if admit:
            lv.lv_whatif_admit(ctx, model, b, p, c, d_ph, ten, L, B, 0.01, A, T, S, stream=stream)
        else:
            lv.lv_whatif(ctx, model, b, p, c, d_ph, T, S, stream=stream)

    d_ph = d(ph)
    _replay(call, [T, S] + ([A] if admit else []), ctx, lv)
