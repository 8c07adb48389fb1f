"""The work that a program built on this library has it do, as cases that can be timed and compared.

One pass is one use of the library through its public calls: a serving step attributed inside a scheduler's loop, a
log of past batches attributed and billed, its features taken out, stored shares added up per tenant, the latency
model fitted and judged, a pending queue tried against candidate batches.

A program keeps one context for its life and one accumulator per billing period, and its output buffers; the model's
coefficients are fixed, the requests are not.  So a case fixes the model, and the seed draws the requests.
"""

import math

import numpy as np
import torch

import paper_2608_08382_gb300 as lv

# Architecture integers of the 8B-class shape whose physical features are taken.
ARCH = (32, 4096, 32, 8, 128, 14336, 2, 2, 1)
SPLIT = (256, 256)

# Cost scales of a served model: bytes of weights a step reads, FLOPs per new token, KV bytes per context token,
# attention FLOPs per squared new token; on 8e12 bytes/s and 1.88e15 FLOP/s.
COSTS = {
    "chat": (13_958_643_712, 13_958_643_712, 131_072, 262_144),
    "continuous": (13_212_057_600, 13_212_057_600, 98_304, 245_760),
    "skew": (13_958_643_712, 13_958_643_712, 131_072, 262_144),
    "planning": (15_602_810_880, 15_602_810_880, 65_536, 163_840),
}

# The request laws: batch sizes, prefills and contexts.
#   chat        20 % prefills of lognormal length on an empty cache, contexts uniform
#   continuous  continuous batching: 0 to 4 chunked prefills of 512 tokens per batch, contexts lognormal
#   skew        heavy-tailed batch sizes (Pareto 1.5), 10 % prefills, lengths log-uniform over five decades
#   planning    30 % prefills, lengths and contexts lognormal with a long tail


def listed():
    return [
        # a scheduler attributes the step it has just run: a small decode-only step, where latency is all there is
        dict(name="step-decode-128", kind="step", n_req=128, prefills=0, n_batch=1, tenants=256),
        # the same call on the largest step of a serving engine: 2,048 sequences with four chunked prefills
        dict(name="step-mixed-2048", kind="step", n_req=2048, prefills=4, n_batch=1, tenants=256),
        # an hour's log of one replica, billed to a few tenants
        dict(name="log-chat-20k", kind="log", law="chat", n_batch=20_000, tenants=16, dtype="f64"),
        # a cluster's log of continuous batches, billed to 256 tenants of uneven size
        dict(name="log-continuous-1m", kind="log", law="continuous", n_batch=1_000_000, tenants=256, dtype="f64"),
        # many tiny batches and a few huge ones, billed to 65,536 tenants
        dict(name="log-skew-10m", kind="log", law="skew", n_batch=10_000_000, tenants=65_536, dtype="f64"),
        # the single-precision variant, for dashboards
        dict(name="log-continuous-f32-300k", kind="log", law="continuous", n_batch=300_000, tenants=256, dtype="f32"),
        # features of every request and batch, then Eq. 1 from the stored sums
        dict(name="features-400k", kind="features", law="chat", n_batch=400_000),
        # shares stored earlier, added up per tenant
        dict(name="accumulate-30m", kind="accumulate", n_req=30_000_001, tenants=3000),
        # the coefficients from two million profiled batches, two latency vectors (two runs of the same batches)
        dict(name="fit-2m", kind="fit", n_batch=2_000_000, size=256, n_y=2),
        # how well predictions met measured latencies
        dict(name="accuracy-2m", kind="accuracy", n=2_000_000),
        # planning: every pending request against every candidate batch
        dict(name="whatif-4096x1024", kind="whatif", pending=4096, cand=1024, tenants=0),
        # admission control between two steps: a short queue, a handful of batches, budgets and a latency objective
        dict(name="admit-500x24", kind="whatif", pending=500, cand=24, tenants=64),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "log", "log", "log", "features", "accumulate", "fit", "accuracy", "whatif"])
    if kind == "step":
        n = _log_int(rng, 16, 4096)
        return dict(kind=kind, n_req=n, prefills=rng.randint(0, min(8, n)), n_batch=rng.choice([1, 1, 2, 5]),
                    tenants=rng.choice([16, 100, 256, 512]))
    if kind == "log":
        law = rng.choice(["chat", "continuous", "skew"])
        most = {"chat": 3_000_000, "continuous": 900_000, "skew": 9_000_000}[law]
        return dict(kind=kind, law=law, n_batch=_log_int(rng, 300, most),
                    tenants=rng.choice([0, 16, 256, 3000, 65_536]), dtype=rng.choice(["f64", "f64", "f32"]))
    if kind == "features":
        return dict(kind=kind, law=rng.choice(["chat", "continuous", "skew"]), n_batch=_log_int(rng, 300, 700_000))
    if kind == "accumulate":
        return dict(kind=kind, n_req=_log_int(rng, 10_000, 100_000_000), tenants=rng.choice([16, 256, 3000, 65_536]))
    if kind == "fit":
        return dict(kind=kind, n_batch=_log_int(rng, 20_000, 1_500_000), size=rng.choice([64, 256]),
                    n_y=rng.randint(1, 4))
    if kind == "accuracy":
        return dict(kind=kind, n=_log_int(rng, 1000, 8_000_000))
    return dict(kind=kind, pending=_log_int(rng, 16, 8192), cand=_log_int(rng, 5, 2048),
                tenants=rng.choice([0, 16, 64]))


# ------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _coef(law):
    """Coefficients [phase * 2 + regime][beta, a1, a2, a3, a4] of the served model: memory-bound segments pay the
    weight load in beta and little per token, compute-bound ones the reverse."""
    weights, flop, kv, attn = COSTS[law]
    rng = np.random.default_rng(20260382)
    c = np.empty((4, 5))
    for s in range(4):
        if s & 1 == 0:
            base = (weights / 8e12, 0.05 * flop / 1.88e15, kv / 8e12, attn / 1.88e15, 1e-8)
        else:
            base = (0.3 * weights / 8e12, flop / 1.88e15, kv / 8e12, attn / 1.88e15, 1e-8)
        c[s] = np.asarray(base) * np.exp(0.2 * rng.standard_normal(5))
    return c


def _randint(g, n, lo, hi):
    """int32 uniform on lo..hi."""
    return torch.randint(lo, hi + 1, (n,), generator=g, device="cuda", dtype=torch.int32)


def _lognormal(g, n, mu, sigma, hi):
    x = torch.empty(n, dtype=torch.float32, device="cuda").log_normal_(mu, sigma, generator=g)
    return x.round_().clamp_(1, hi).to(torch.int32)


def _log_uniform(g, n, hi):
    x = torch.rand(n, generator=g, device="cuda").mul_(math.log(hi)).exp_().floor_()
    return x.clamp_(1, hi).to(torch.int32)


def _zipf(g, n, tenants, s):
    """Tenant ids, id k - 1 as often as k^-s."""
    w = torch.arange(1, tenants + 1, dtype=torch.float64, device="cuda") ** -s
    cdf = (torch.cumsum(w, 0) / w.sum()).to(torch.float32)
    out = torch.empty(n, dtype=torch.int32, device="cuda")
    for i in range(0, n, 1 << 25):
        u = torch.rand(min(1 << 25, n - i), generator=g, device="cuda")
        out[i:i + u.numel()] = torch.searchsorted(cdf, u, right=True, out_int32=True).clamp_(max=tenants - 1)
    return out


def _sizes(g, law, n_batch, size):
    """Requests per batch: the same sizes for every seed, in the seed's order, so that a case has one number of
    requests."""
    fixed = _generator(20260382)
    if law == "skew":
        u = 1.0 - torch.rand(n_batch, generator=fixed, device="cuda", dtype=torch.float64)
        sizes = u.pow_(-1 / 1.5).floor_().clamp_(1, 4096).to(torch.int64)
    else:
        lo, hi = {"chat": (1, size or 64), "continuous": (16, 256), "planning": (32, 256)}[law]
        sizes = torch.randint(lo, hi + 1, (n_batch,), generator=fixed, device="cuda")
    return sizes[torch.randperm(n_batch, generator=g, device="cuda")]


def _requests(g, law, n_batch, tenants, size=0, c_hi=8192):
    off = torch.zeros(n_batch + 1, dtype=torch.int64, device="cuda")
    sizes = _sizes(g, law, n_batch, size)
    torch.cumsum(sizes, 0, out=off[1:])
    n = int(off[-1])
    if law == "continuous":
        phase = torch.zeros(n, dtype=torch.int32, device="cuda")
        k = torch.randint(0, 5, (n_batch,), generator=g, device="cuda")
        for j in range(4):
            at = off[:-1] + (torch.rand(n_batch, generator=g, device="cuda", dtype=torch.float64) * sizes).to(torch.int64)
            phase[at[k > j]] = 1
        pre = phase == 1
        p = torch.where(pre, 512, 1).to(torch.int32)
        c = torch.where(pre, _randint(g, n, 0, 32256), _lognormal(g, n, 7.5, 1.2, 32768))
        s = 1.1
    else:
        prob = {"chat": 0.2, "skew": 0.1, "planning": 0.3}[law]
        pre = torch.rand(n, generator=g, device="cuda") < prob
        phase = pre.to(torch.int32)
        if law == "chat":
            new, ctx, s = _lognormal(g, n, 6.0, 1.0, 8192), _randint(g, n, 1, c_hi), 0.0
        elif law == "skew":
            new, ctx, s = _log_uniform(g, n, 16384), _log_uniform(g, n, 131_072), 1.2
        else:
            new, ctx, s = _lognormal(g, n, 8.0, 1.3, 131_072), _lognormal(g, n, 8.0, 1.3, 131_072), 0.0
        one = torch.ones((), dtype=torch.int32, device="cuda")
        p, c = torch.where(pre, new, one), torch.where(pre, torch.zeros_like(one), ctx)
    t = _zipf(g, n, tenants, s) if tenants else None
    return lv.Batches(p=p, c=c, phase=phase, offsets=off, tenant=t, n_tenants=tenants)


def _step_requests(g, case):
    """One step's batches: decodes with the given number of chunked prefills among them."""
    n, nb = case["n_req"], case["n_batch"]
    phase = torch.zeros(n, dtype=torch.int32, device="cuda")
    phase[torch.randperm(n, generator=g, device="cuda")[:case["prefills"]]] = 1
    pre = phase == 1
    p = torch.where(pre, 512, 1).to(torch.int32)
    c = torch.where(pre, _randint(g, n, 0, 32256), _lognormal(g, n, 7.5, 1.2, 32768))
    off = torch.tensor([n * b // nb for b in range(nb + 1)], dtype=torch.int64, device="cuda")
    return lv.Batches(p=p, c=c, phase=phase, offsets=off, tenant=_zipf(g, n, case["tenants"], 1.1),
                      n_tenants=case["tenants"])


def _sums(b):
    """Per batch S1, S2, S3, n and the segment, exact integers."""
    def total(x):
        z = torch.zeros(x.numel() + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(x, 0, out=z[1:])
        return z[b.offsets[1:]] - z[b.offsets[:-1]]

    p = b.p.to(torch.int64)
    s1, s3 = total(p), total(p * p)
    s2 = total(b.c.to(torch.int64))
    pre = total(b.phase.to(torch.int64)) > 0
    n = b.offsets[1:] - b.offsets[:-1]
    split = torch.where(pre, SPLIT[1], SPLIT[0])
    return s1, s2, s3, n, pre.to(torch.int64) * 2 + (s1 >= split).to(torch.int64)


def _eq1(k, s1, s2, s3, n):
    k0, k1, k2, k3, k4 = k.unbind(-1)
    return k0 + k1 * s1 + k2 * s2 + k3 * s3 + k4 * (n * n)


def _data(case, seed):
    """The case's inputs, from the seed alone."""
    g = _generator(seed)
    kind = case["kind"]
    if kind == "step":
        return dict(b=_step_requests(g, case), law="continuous")
    if kind == "log":
        return dict(b=_requests(g, case["law"], case["n_batch"], case["tenants"]), law=case["law"])
    if kind == "features":
        return dict(b=_requests(g, case["law"], case["n_batch"], 0), law=case["law"])
    if kind == "accumulate":
        share = torch.empty(case["n_req"], dtype=torch.float64, device="cuda").log_normal_(-11.0, 1.0, generator=g)
        return dict(share=share, tenant=_zipf(g, case["n_req"], case["tenants"], 1.1))
    if kind == "fit":
        # latencies: the model's own with a few percent of measurement noise
        b = _requests(g, "chat", case["n_batch"], 0, size=case["size"], c_hi=16384)
        s1, s2, s3, n, seg = _sums(b)
        T = _eq1(torch.tensor(_coef("chat"), device="cuda")[seg], s1, s2, s3, n)
        z = torch.randn(case["n_y"], case["n_batch"], generator=g, device="cuda", dtype=torch.float64)
        return dict(b=b, y=T * torch.exp(0.03 * z))
    if kind == "accuracy":
        T = torch.rand(case["n"], generator=g, device="cuda", dtype=torch.float64).mul_(4.0).exp_().mul_(2e-3)
        z = torch.randn(case["n"], generator=g, device="cuda", dtype=torch.float64)
        return dict(T=T, y=T * torch.exp(0.03 * z))
    cand = _requests(g, "planning", case["cand"], 0)
    np_ = case["pending"]
    ph = (torch.rand(np_, generator=g, device="cuda") < 0.3).to(torch.int32)
    p = torch.where(ph == 1, _lognormal(g, np_, 8.0, 1.3, 131_072), 1).to(torch.int32)
    c = torch.where(ph == 1, 0, _lognormal(g, np_, 8.0, 1.3, 131_072)).to(torch.int32)
    d = dict(b=cand, p=p, c=c, ph=ph, law="planning")
    if case["tenants"]:
        d["tenant"] = torch.randint(0, case["tenants"], (np_,), generator=g, device="cuda", dtype=torch.int32)
        d["L"] = torch.rand(case["tenants"], generator=g, device="cuda", dtype=torch.float64).mul_(2e-3)
        d["budget"] = torch.full((case["tenants"],), 4e-3, dtype=torch.float64, device="cuda")
        d["slo"] = 0.06
    return d


_kept = []


def _context():
    """The process's context."""
    if not _kept:
        _kept.append(lv.Context())
    return _kept[0]


def prepare(case, seed):
    s = _data(case, seed)
    s["case"], s["ctx"] = dict(case), _context()
    kind = case["kind"]
    if "law" in s:
        s["model"] = lv.make_model(_coef(s["law"]), SPLIT)

    def out(*shape, dtype=torch.float64):
        return torch.empty(*shape, dtype=dtype, device="cuda")

    if kind in ("step", "log"):
        dt = torch.float32 if case.get("dtype") == "f32" else torch.float64
        s["T"], s["share_out"] = out(s["b"].n_batch, dtype=dt), out(s["b"].n_req, dtype=dt)
    if kind in ("step", "log", "accumulate") and case["tenants"]:
        s["acc"], s["L"] = lv.TenantAcc(s["ctx"], case["tenants"]), out(case["tenants"])
    if kind == "features":
        b = s["b"]
        s["req"], s["feat"] = out(3, b.n_req, dtype=torch.int64), out(5, b.n_batch, dtype=torch.int64)
        s["seg"], s["T"] = out(b.n_batch, dtype=torch.uint8), out(b.n_batch)
    if kind == "whatif":
        shape = (case["pending"], case["cand"])
        s["T"], s["share_out"] = out(*shape), out(*shape)
        if case["tenants"]:
            s["admit"] = out(*shape, dtype=torch.uint8)
    return s


# ------------------------------------------------------------------ one pass

def run(s):
    kind, ctx = s["case"]["kind"], s["ctx"]
    if kind == "step":
        lv.lv_attribute_step(ctx, s["model"], s["b"], s["T"], s["share_out"], s["acc"], s["L"], reset=True)
        return dict(T=s["T"], share=s["share_out"], L=s["L"])
    if kind == "log":
        call = lv.lv_attribute_f32 if s["case"]["dtype"] == "f32" else lv.lv_attribute
        if "acc" not in s:
            call(ctx, s["model"], s["b"], s["T"], s["share_out"])
            return dict(T=s["T"], share=s["share_out"])
        s["acc"].reset()
        call(ctx, s["model"], s["b"], s["T"], s["share_out"], s["acc"])
        lv.lv_tenant_totals(ctx, s["acc"], s["L"])
        return dict(T=s["T"], share=s["share_out"], L=s["L"])
    if kind == "features":
        lv.lv_features(ctx, s["b"], ARCH, s["model"], s["req"], s["feat"], s["seg"])
        lv.lv_batch_latency(ctx, s["model"], s["feat"], s["seg"], s["T"])
        return dict(req=s["req"], feat=s["feat"], seg=s["seg"], T=s["T"])
    if kind == "accumulate":
        s["acc"].reset()
        lv.lv_tenant_accumulate(ctx, s["acc"], s["share"], s["tenant"])
        lv.lv_tenant_totals(ctx, s["acc"], s["L"])
        return dict(L=s["L"])
    if kind == "fit":
        models = [lv.make_model(np.zeros((4, 5)), SPLIT) for _ in range(s["case"]["n_y"])]
        rep = lv.lv_fit(ctx, s["b"], s["y"], models)
        c = np.stack([lv.model_coef(m) for m in models])
        return dict(beta=c[:, :, 0], a1=c[:, :, 1], a2=c[:, :, 2], a3=c[:, :, 3], a4=c[:, :, 4],
                    n=np.array([r["n"] for r in rep]), status=np.array([r["status"] for r in rep]),
                    dropped=np.array([r["dropped"] for r in rep]), ssr=np.array([r["ssr"] for r in rep]),
                    r2=np.array([r["r2"] for r in rep]))
    if kind == "accuracy":
        return lv.lv_accuracy(ctx, s["y"], s["T"])
    if "admit" in s:
        lv.lv_whatif_admit(ctx, s["model"], s["b"], s["p"], s["c"], s["ph"], s["tenant"], s["L"], s["budget"],
                           s["slo"], s["admit"], s["T"], s["share_out"])
        return dict(T=s["T"], share=s["share_out"], admit=s["admit"])
    lv.lv_whatif(ctx, s["model"], s["b"], s["p"], s["c"], s["ph"], s["T"], s["share_out"])
    return dict(T=s["T"], share=s["share_out"])


# ------------------------------------------------------------------ what a pass cannot do without

_MEAN = {"chat": 32.5, "continuous": 136.0, "skew": 2.6, "planning": 144.0}  # requests per batch


def work(case):
    """Each input read once, each output written once; the operations of Eq. 1 and the shares."""
    kind = case["kind"]
    if kind == "step":
        r, nb, t = case["n_req"], case["n_batch"], case["tenants"]
        return dict(bytes=24.0 * r + 16 * nb + 8 * t, flops=8.0 * r)
    if kind == "log":
        nb, t = case["n_batch"], case["tenants"]
        r = nb * _MEAN[case["law"]]
        wide = 4 if case["dtype"] == "f32" else 8
        return dict(bytes=(12.0 + wide + (4 if t else 0)) * r + (8 + wide) * nb + 8 * t, flops=10.0 * r + 8 * nb)
    if kind == "features":
        nb = case["n_batch"]
        r = nb * _MEAN[case["law"]]
        return dict(bytes=(12.0 + 24) * r + (8 + 41 + 8) * nb, flops=8.0 * r + 8 * nb)
    if kind == "accumulate":
        return dict(bytes=12.0 * case["n_req"] + 8 * case["tenants"], flops=1.0 * case["n_req"])
    if kind == "fit":
        nb = case["n_batch"]
        r = nb * (case["size"] + 1) / 2
        return dict(bytes=12.0 * r + (8 + 8 * case["n_y"]) * nb, flops=5.0 * r + (30 + 12 * case["n_y"]) * nb)
    if kind == "accuracy":
        return dict(bytes=16.0 * case["n"], flops=12.0 * case["n"])
    pairs = case["pending"] * case["cand"]
    cand = case["cand"] * _MEAN["planning"]
    return dict(bytes=(16.0 + (1 if case["tenants"] else 0)) * pairs + 12 * cand + 12 * case["pending"],
                flops=10.0 * pairs)


def tolerance(case):
    """Relative error that a correct implementation at the same precision shows.  The sums of a batch are exact
    integers and 64-bit results are rounded once or a few times; the fitted coefficients carry the conditioning of
    the normal equations."""
    kind = case["kind"]
    if kind == "fit":
        return dict(rel=1e-12, max=1e-11)
    if kind == "accuracy":
        return dict(rel=1e-12, max=1e-12)
    if kind == "log" and case["dtype"] == "f32":
        return dict(rel=3e-7, max=1e-6)
    if kind in ("log", "accumulate"):  # up to 1e8 shares per tenant, in any order
        return dict(rel=1e-12, max=1e-11)
    # whole values: admission bits of pairs that lie on a bound (the features are exact)
    return dict(rel=2e-15, max=1e-14, differ=1e-6 if kind == "whatif" else 0.0)


# ------------------------------------------------------------------ the same in plain 64-bit torch

def _fit_exact(s, case):
    s1, s2, s3, n, seg = _sums(s["b"])
    n_y = case["n_y"]
    coef = np.zeros((n_y, 4, 5))
    ssr, r2 = np.zeros((n_y, 4)), np.zeros((n_y, 4))
    X = torch.stack([torch.ones_like(s1), s1, s2, s3, n * n], 1).to(torch.float64)
    for g in range(4):
        m = seg == g
        x = X[m]
        cols = [0, 1, 2, 3, 4] if bool((x[:, 1] != x[:, 3]).any()) else [0, 1, 2, 4]
        if x.shape[0] < len(cols):
            continue
        scale = x[:, cols].abs().amax(0)
        q, r = torch.linalg.qr(x[:, cols] / scale)
        for k in range(n_y):
            y = s["y"][k][m]
            w = torch.linalg.solve_triangular(r, (q.T @ y)[:, None], upper=True)[:, 0] / scale
            res = y - x[:, cols] @ w
            coef[k, g, cols] = w.cpu().numpy()
            ssr[k, g] = float((res * res).sum())
            r2[k, g] = 1 - ssr[k, g] / float(((y - y.mean()) ** 2).sum())
    return dict(beta=coef[:, :, 0], a1=coef[:, :, 1], a2=coef[:, :, 2], a3=coef[:, :, 3], a4=coef[:, :, 4], n=None,
                status=None, dropped=None, ssr=ssr, r2=r2)


def exact(case, seed):
    s = _data(case, seed)
    kind = case["kind"]
    if kind == "fit":
        return _fit_exact(s, case)
    if kind == "accumulate":
        return dict(L=torch.bincount(s["tenant"], weights=s["share"], minlength=case["tenants"]))
    if kind == "accuracy":
        y, T = s["y"], s["T"]
        rel = ((T - y).abs() / y).sort().values
        dy, dT = y - y.mean(), T - T.mean()
        at = [float(rel[max(1, math.ceil(q * y.numel() / 100)) - 1]) for q in (50, 90, 99)]
        return dict(n=None, r2_ssr=float(1 - ((y - T) ** 2).sum() / (dy * dy).sum()),
                    r2_corr=float((dy * dT).sum() ** 2 / ((dy * dy).sum() * (dT * dT).sum())),
                    mean_rel=float(rel.mean()), p50=at[0], p90=at[1], p99=at[2])
    k = torch.tensor(_coef(s["law"]), device="cuda")
    b = s["b"]
    s1, s2, s3, n, seg = _sums(b)
    if kind == "whatif":
        pre = (seg[None, :] >= 2) | (s["ph"][:, None] == 1)
        p, c = s["p"].to(torch.int64)[:, None], s["c"].to(torch.int64)[:, None]
        t1 = s1[None, :] + p
        kk = k[pre.to(torch.int64) * 2 + (t1 >= torch.where(pre, SPLIT[1], SPLIT[0])).to(torch.int64)]
        n1 = n[None, :] + 1
        T = _eq1(kk, t1, s2[None, :] + c, s3[None, :] + p * p, n1)
        share = kk[..., 0] / n1 + kk[..., 1] * p + kk[..., 2] * c + kk[..., 3] * (p * p) + kk[..., 4] * n1
        return dict(T=T, share=share, admit=None)
    T = _eq1(k[seg], s1, s2, s3, n)
    if kind == "features":
        return dict(req=None, feat=None, seg=None, T=T)
    r = torch.repeat_interleave(torch.arange(b.n_batch, device="cuda"), n)
    kk = k[seg]
    const = (kk[:, 0] / n + kk[:, 4] * n)[r]
    slopes, which = k[:, 1:4].T.contiguous(), seg[r]
    p, c = b.p.to(torch.float64), b.c.to(torch.float64)
    share = const + slopes[0][which] * p + slopes[1][which] * c + slopes[2][which] * (p * p)
    if not case["tenants"]:
        return dict(T=T, share=share)
    return dict(T=T, share=share, L=torch.bincount(b.tenant, weights=share, minlength=case["tenants"]))
