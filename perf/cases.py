"""The calls whose time this repository keeps an eye on.

Each case is one call (or the few calls of one step) that a user of the
library makes through ``paper_1308_2572_gb300.art`` or ``.autograd``: pricing
one layer, running a portfolio of layers, the all-FP64 form, the metrics of a
finished YLT, per-event payouts, sensitivities, and the path from host
buffers. Sizes follow the workloads of ``workloads.py`` (c0 to c4); inputs
are drawn on the device from a seed with that module's distributions.

A case is a dict of plain values:
  kind       which call (see ``run``)
  catalogue, elts, nnz_lo, nnz_hi, mu, sigma
             the ELT pool: ``elts`` tables over ``catalogue`` events, each with
             nnz_lo .. nnz_hi expected non-zero lognormal(mu, sigma) losses
  layers, per_lo, per_hi
             layers of per_lo .. per_hi distinct ELTs of the pool (per_lo = 0:
             layer j covers ELTs (2 j + i) mod elts for i < per_hi)
  spread     occurrence terms drawn per layer (else 1e5 / 5e6 for all)
  unlimited  every second layer has an unlimited occurrence cover
  trials, events, ragged
             the YET: ``events`` per trial, or Poisson lengths as a CSR
  probs      1 or 3 probabilities
"""
import numpy as np
import torch
import torch.nn.functional as F

from paper_1308_2572_gb300 import art, autograd

PROBS = {1: [0.99], 3: [0.99, 0.996, 0.999]}


def _case(name, kind, **kw):
    c = dict(kind=kind, catalogue=2_000_000, elts=16, nnz_lo=20_000, nnz_hi=20_000, mu=12.0, sigma=2.0, layers=1,
             per_lo=0, per_hi=16, spread=False, unlimited=False, trials=1_000_000, events=1000, ragged=False, probs=1)
    c.update(kw)
    if name:
        c = dict(name=name, **c)
    return c


_C2 = dict(elts=256, nnz_lo=10_000, nnz_hi=50_000, sigma=2.5, per_lo=1, per_hi=32, spread=True)
_C4 = dict(elts=512, nnz_lo=10_000, nnz_hi=50_000, mu=13.0, sigma=2.5, per_lo=4, per_hi=32, spread=True, probs=3)


def listed():
    return [
        # a quick quote: one small layer over a regional catalogue, few trials (c0's portfolio; launches count)
        _case("quote_small", "price", catalogue=100_000, elts=3, nnz_lo=10_000, nnz_hi=10_000, per_hi=3, trials=1_000),
        # pricing one layer against an ordinary YET of ragged trials, the metrics included
        _case("price_layer", "price", trials=50_003, ragged=True),
        # the paper's headline run: 1e6 trials x 1000 events x 16 ELTs (c1), as the benchmark sets it up
        _case("layer_1m", "forward"),
        # a 64-layer book over ragged trials with the library's defaults (c2)
        _case("book_64", "forward_default", layers=64, trials=100_001, ragged=True, **_C2),
        # the largest run: 128 layers over 512 ELTs, a million trials (c4)
        _case("book_128_1m", "forward", layers=128, **_C4),
        # the all-FP64 form on part of that book, for results that need it
        _case("book_fp64", "forward64", layers=16, trials=100_000, **_C4),
        # a pricing loop's step: EL and TVaR of 8 layers and their gradients with respect to all terms (c3)
        _case("sensitivity", "sensitivity", layers=8, per_hi=8, trials=500_000),
        # the adjoint over layers of many ELTs and ragged trials, for a caller's own weights per trial
        _case("adjoint_wide", "adjoint", layers=12, trials=50_000, ragged=True, **_C2),
        # the metrics of one layer's YLT (the second half of the headline step)
        _case("metrics_layer", "metrics"),
        # the metrics of a whole book's YLT at three return periods
        _case("metrics_book", "metrics", layers=128, probs=3),
        # per-event payouts of one layer (which events pay, which one exhausts the cover)
        _case("payouts", "payouts", trials=100_000),
        # the whole call from pinned host buffers: one layer, YET read over the host link, metrics back
        _case("from_host", "host", trials=100_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["price", "price", "forward", "forward", "forward", "forward_default", "forward64", "sensitivity",
                       "adjoint", "metrics", "metrics", "payouts", "host"])
    if kind == "metrics":
        layers = _log_int(rng, 1, 128)
        return _case(None, kind, layers=layers, trials=_log_int(rng, 5_000, 1_000_000), probs=rng.choice([1, 3]))
    events = _log_int(rng, 200, 1500)
    ragged = rng.random() < 0.5
    kw = dict(catalogue=_log_int(rng, 100_000, 2_000_000), events=events, ragged=ragged, unlimited=rng.random() < 0.15)
    top = min(1_000_000, 1_000_000_000 // events)
    if kind in ("price", "payouts", "host"):
        n = rng.randint(1, 32)
        frac = rng.uniform(0.005, 0.05)
        nnz = max(1, int(frac * kw["catalogue"]))
        cap = {"price": top, "payouts": top // 8, "host": top // 8}[kind]
        return _case(None, kind, elts=n, per_hi=n, nnz_lo=nnz, nnz_hi=nnz, trials=_log_int(rng, 500, cap), **kw)
    if kind == "sensitivity":
        n = rng.choice([8, 16])
        kw.update(elts=n, per_hi=n // 2, layers=rng.randint(1, 8), trials=_log_int(rng, 2_000, top // 2))
        kw.update(nnz_lo=kw["catalogue"] // 100, nnz_hi=kw["catalogue"] // 100)
        return _case(None, kind, **kw)
    base = dict(_C2 if rng.random() < 0.5 else _C4)
    base.update(nnz_lo=kw["catalogue"] // 200, nnz_hi=kw["catalogue"] // 40)
    if kind == "adjoint":
        return _case(None, kind, layers=rng.randint(1, 16), trials=_log_int(rng, 2_000, top // 16), **dict(base, **kw))
    if kind == "forward64":
        return _case(None, kind, layers=_log_int(rng, 1, 32), trials=_log_int(rng, 2_000, top // 4), **dict(base, **kw))
    if kind == "forward_default":
        return _case(None, kind, layers=_log_int(rng, 2, 64), trials=_log_int(rng, 2_000, top // 4), **dict(base, **kw))
    return _case(None, kind, layers=_log_int(rng, 1, 128), trials=_log_int(rng, 2_000, top), **dict(base, **kw))


# ------------------------------------------------------------------ inputs

class _Inputs:
    pass


def _inputs(case, seed):
    """ELT losses, terms and YET of a case, from the seed alone."""
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(seed)
    r = np.random.Generator(np.random.PCG64(seed))
    x = _Inputs()
    C, E, L = case["catalogue"], case["elts"], case["layers"]
    nnz = r.integers(case["nnz_lo"], case["nnz_hi"] + 1, size=E)
    x.losses = torch.zeros((E, C), dtype=torch.float32, device=dev)
    ded, lim = np.empty(E, np.float32), np.empty(E, np.float32)
    q = torch.tensor([0.05, 0.99], dtype=torch.float64, device=dev)
    terms = torch.empty((E, 2), dtype=torch.float64, device=dev)
    for e in range(E):
        row = x.losses[e]
        hit = torch.rand(C, generator=g, device=dev) < float(nnz[e]) / C
        hit[e % C] = True  # an ELT is never empty
        at = hit.nonzero()[:, 0]
        v = torch.exp(case["mu"] + case["sigma"] * torch.randn(at.numel(), generator=g, device=dev))
        row[at] = v
        terms[e] = torch.quantile(v.double(), q)
    t = terms.cpu().numpy()
    ded[:], lim[:] = t[:, 0], t[:, 1]
    x.ded, x.lim = ded, lim
    x.mult = r.uniform(0.9, 1.1, size=E).astype(np.float32)
    if case["per_lo"]:
        sizes = r.integers(case["per_lo"], case["per_hi"] + 1, size=L)
        x.lists = [np.sort(r.choice(E, size=int(s), replace=False)).astype(np.int32) for s in sizes]
    else:
        x.lists = [np.array([(2 * j + i) % E for i in range(case["per_hi"])], dtype=np.int32) for j in range(L)]
    x.off = np.concatenate([[0], np.cumsum([len(l) for l in x.lists])]).astype(np.int32)
    hits = np.array([nnz[l].sum() for l in x.lists]) / C * case["events"]
    scale = 3.0 if case["mu"] > 12.5 else 1.0
    x.terms = np.empty((L, 4))
    if case["spread"]:
        x.terms[:, 0] = np.exp(r.uniform(np.log(1e5), np.log(1e6), size=L))
        x.terms[:, 1] = x.terms[:, 0] * np.exp(r.uniform(np.log(10.0), np.log(100.0), size=L))
    else:
        x.terms[:, 0], x.terms[:, 1] = 1e5, 5e6
    x.terms[:, 2] = hits * scale * np.exp(r.uniform(np.log(1.2e5), np.log(9e5), size=L))
    x.terms[:, 3] = x.terms[:, 2] * np.exp(r.uniform(np.log(0.5), np.log(3.0), size=L))
    x.terms[:, :2] = x.terms[:, :2].astype(np.float32)
    if case["unlimited"]:
        x.terms[1::2, 1] = np.inf
        x.terms[0, 1] = np.inf if L == 1 else x.terms[0, 1]
    T, K = case["trials"], case["events"]
    x.trials = T
    x.k = K
    x.trial_off = None
    total = T * K
    if case["ragged"]:
        n = torch.poisson(torch.full((T,), float(K), device=dev), generator=g).clamp_(K // 5, 2 * K).to(torch.int64)
        x.trial_off = torch.zeros(T + 1, dtype=torch.int64, device=dev)
        torch.cumsum(n, 0, out=x.trial_off[1:])
        total = int(x.trial_off[-1])
        x.k = 0
    x.ids = torch.randint(0, C, (total,), generator=g, device=dev, dtype=torch.int32)
    return x


def _ylt_inputs(case, seed):
    """A YLT as a book leaves it: per layer some trials without a loss, some
    at the aggregate cap, the rest skewed in between."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    L, T = case["layers"], case["trials"]
    ylt = torch.empty((L, T), dtype=torch.float64, device="cuda")
    r = np.random.Generator(np.random.PCG64(seed))
    for j in range(L):
        ret, cap = r.uniform(-1.0, 0.8), r.uniform(0.8, 3.0)
        s = torch.randn(T, generator=g, device="cuda", dtype=torch.float64)
        ylt[j] = 1e8 * (torch.exp(0.5 * s) - np.exp(0.5 * ret)).clamp_(0.0, cap)
    return ylt


def _probs(case):
    return PROBS[case["probs"]]


def _portfolio(x, **kw):
    return art.art_create_portfolio(x.losses.shape[1], x.losses, x.mult, x.ded, x.lim, x.off, np.concatenate(x.lists),
                                    x.terms, **kw)


def prepare(case, seed):
    kind = case["kind"]
    s = _Inputs()
    s.case, s.kind = case, kind
    s.probs = _probs(case)
    L, T, n_p = case["layers"], case["trials"], len(s.probs)
    f64 = dict(dtype=torch.float64, device="cuda")
    if kind in ("price", "metrics"):
        s.mean = torch.empty(L, **f64)
        s.pml = torch.empty((L, n_p), **f64)
        s.tvar = torch.empty((L, n_p), **f64)
    if kind == "metrics":
        s.ylt = _ylt_inputs(case, seed)
        return s
    x = _inputs(case, seed)
    layer_csr = art.ART_LAYOUT_LAYER | art.ART_LAYOUT_SPARSE
    if kind == "forward":
        # the fastest variant and the persisting L2 window, as the benchmark runs
        s.p = _portfolio(x, layouts=layer_csr, variant=art.ART_VARIANT_SKIP, flags=art.ART_FLAG_L2_PERSIST)
    elif kind == "forward64":
        s.p = _portfolio(x, layouts=layer_csr | art.ART_LAYOUT_OCC64, variant=art.ART_VARIANT_FP64)
    elif kind == "adjoint":
        s.p = _portfolio(x, layouts=layer_csr | art.ART_LAYOUT_GROUP, variant=art.ART_VARIANT_SKIP)
    else:
        s.p = _portfolio(x)
    if kind == "host":
        s.ids = torch.empty(x.ids.numel(), dtype=torch.int32, pin_memory=True)
        s.ids.copy_(x.ids)
        s.off = None
        if x.trial_off is not None:
            s.off = torch.empty(T + 1, dtype=torch.int64, pin_memory=True)
            s.off.copy_(x.trial_off)
        s.mean = torch.empty(L, dtype=torch.float64)
        s.pml = torch.empty((L, n_p), dtype=torch.float64)
        s.tvar = torch.empty((L, n_p), dtype=torch.float64)
    else:
        s.ids, s.off = x.ids, x.trial_off
    s.k = x.k
    if kind in ("price", "forward", "forward_default", "forward64", "adjoint"):
        s.ylt = torch.empty((L, T), **f64)
    if kind == "payouts":
        s.pay = torch.empty(x.ids.numel(), **f64)
        s.exhaust = torch.empty(T, dtype=torch.int32, device="cuda")
        s.ylt = torch.empty(T, **f64)
    if kind == "adjoint":
        s.branch = torch.empty((L, T), dtype=torch.uint8, device="cuda")
        s.weights = _weights(case, seed)
        s.g_terms = torch.empty((L, 4), **f64)
        s.g_mult = torch.empty(case["elts"], **f64)
    if kind == "sensitivity":
        s.leaves = [torch.tensor(np.ascontiguousarray(x.terms[:, i]), requires_grad=True) for i in range(4)]
        s.leaves.append(torch.tensor(x.mult.astype(np.float64), requires_grad=True))
        s.g_out = [torch.full((L,), 1.0, dtype=torch.float64), torch.full((L, n_p), 0.25, dtype=torch.float64)]
    return s


def _weights(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    return torch.rand((case["layers"], case["trials"]), generator=g, device="cuda", dtype=torch.float64) / case["trials"]


# --------------------------------------------------------------------- run

def run(s):
    L, T = s.case["layers"], s.case["trials"]
    if s.kind == "metrics":
        art.art_metrics(s.ylt, T, L, s.probs, s.mean, s.pml, s.tvar)
        return {"mean": s.mean, "pml": s.pml, "tvar": s.tvar}
    if s.kind == "price":
        art.art_run_ylt(s.p, T, s.ids, s.off, s.k, s.ylt)
        art.art_metrics(s.ylt, T, L, s.probs, s.mean, s.pml, s.tvar)
        return {"ylt": s.ylt, "mean": s.mean, "pml": s.pml, "tvar": s.tvar}
    if s.kind == "payouts":
        art.art_run_payouts(s.p, 0, T, s.ids, s.off, s.k, s.pay, s.exhaust, s.ylt)
        return {"payouts": s.pay, "exhaust": s.exhaust, "ylt": s.ylt}
    if s.kind == "host":
        art.art_run_ylt_host_metrics(s.p, T, s.ids, s.off, s.k, s.probs, mean=s.mean, pml=s.pml, tvar=s.tvar)
        return {"mean": s.mean, "pml": s.pml, "tvar": s.tvar}
    if s.kind == "sensitivity":
        mean, tvar = autograd.layer_metrics(s.p, (s.ids, s.off, s.k, T), s.probs, *s.leaves)
        grads = torch.autograd.grad([mean, tvar], s.leaves, s.g_out)
        return {"mean": mean.detach(), "tvar": tvar.detach(), "occ_ret": grads[0], "occ_lim": grads[1],
                "agg_ret": grads[2], "agg_lim": grads[3], "mult": grads[4]}
    if s.kind == "adjoint":
        art.art_run_ylt(s.p, T, s.ids, s.off, s.k, s.ylt, s.branch)
        art.art_run_ylt_backward(s.p, T, s.ids, s.off, s.k, s.branch, s.weights, s.g_terms, s.g_mult)
        return {"ylt": s.ylt, "branch": s.branch, "terms": s.g_terms, "mult": s.g_mult}
    art.art_run_ylt(s.p, T, s.ids, s.off, s.k, s.ylt)
    return {"ylt": s.ylt}


# -------------------------------------------------------------------- work

def work(case):
    """The ids (and offsets) and each ELT's non-zero losses read once, the
    outputs written once; one addition per event and layer (and per event
    and layer's ELT with a gradient), no more than 1 in the metrics per loss."""
    kind, L, T = case["kind"], case["layers"], case["trials"]
    n_p = len(_probs(case))
    if kind == "metrics":
        return {"bytes": 8 * L * T + 8 * L * (1 + 2 * n_p), "flops": L * T}
    events = T * case["events"]
    nbytes = 4 * events + (8 * (T + 1) if case["ragged"] else 0)
    nbytes += 8 * case["elts"] * (case["nnz_lo"] + case["nnz_hi"]) // 2
    flops = events * L
    if kind == "payouts":
        return {"bytes": nbytes + 8 * events + 12 * T, "flops": 2 * events}
    if kind == "sensitivity":
        return {"bytes": nbytes + 8 * L * 7 + 8 * case["elts"], "flops": 2 * flops}
    if kind == "adjoint":
        return {"bytes": nbytes + 17 * L * T + 32 * L + 8 * case["elts"], "flops": 2 * flops}
    if kind == "host":
        return {"bytes": nbytes + 8 * L * (1 + 2 * n_p), "flops": flops}
    return {"bytes": nbytes + 8 * L * T, "flops": flops}


# ------------------------------------------------------------------- exact

def _bags(x, tables, step_events=1 << 27):
    """Per trial, the sums of the rows of ``tables`` [C][n] its events select."""
    T = x.trials
    n = tables.shape[1]
    out = torch.empty((T, n), dtype=torch.float64, device="cuda")
    off = x.trial_off if x.trial_off is not None else torch.arange(T + 1, device="cuda", dtype=torch.int64) * x.k
    step = max(1, min(T, step_events * T // max(1, x.ids.numel())))
    for t0 in range(0, T, step):
        t1 = min(T, t0 + step)
        b, e = int(off[t0]), int(off[t1])
        if e == b:
            out[t0:t1] = 0.0
            continue
        out[t0:t1] = F.embedding_bag(x.ids[b:e].long(), tables, (off[t0:t1] - b), mode="sum")
    return out


def _fin64(x, e):
    y = x.losses[e].double() * float(x.mult[e]) - float(x.ded[e])
    return y.clamp_(0.0, float(x.lim[e]))


def _event_sums64(x, layers=None):
    """x_j per catalogue event, [C][layers] in FP64."""
    layers = range(len(x.lists)) if layers is None else layers
    out = torch.zeros((x.losses.shape[1], len(layers)), dtype=torch.float64, device="cuda")
    for s, j in enumerate(layers):
        acc = torch.zeros(x.losses.shape[1], dtype=torch.float64, device="cuda")
        for e in x.lists[j]:
            acc += _fin64(x, int(e))
        out[:, s] = acc
    return out


def _xl(v, ret, lim):
    return torch.minimum((v - ret).clamp_(min=0.0), lim)


def _cols(x):
    return [torch.tensor(x.terms[:, i], dtype=torch.float64, device="cuda") for i in range(4)]


def _rank(p, n):
    q = (1.0 - p) * n
    k = round(q) if abs(q - round(q)) <= 1e-9 * n else int(np.ceil(q))
    return min(n, max(1, int(k)))


def _metrics64(ylt, probs):
    top = torch.topk(ylt, _rank(min(probs), ylt.shape[1]), dim=1, sorted=True).values
    ks = [_rank(p, ylt.shape[1]) for p in probs]
    pml = torch.stack([top[:, k - 1] for k in ks], 1)
    tvar = torch.stack([top[:, :k].mean(1) for k in ks], 1)
    return ylt.mean(1), pml, tvar


def _gradients64(x, s_sum, weights, occ_x):
    """Gradients of sum weights * Y with respect to the terms and multipliers."""
    ocr, ocl, agr, agl = _cols(x)
    w = s_sum - agr
    mid = (w > 0) & (w < agl)
    cap = w > agl
    ga = weights.t() * mid
    g_agr = -ga.sum(0)
    g_agl = (weights.t() * cap).sum(0)
    wo = occ_x - ocr
    n_mid = _bags(x, ((wo > 0) & (wo < ocl)).double())
    n_cap = _bags(x, (wo > ocl).double())
    g_ocr = -(ga * n_mid).sum(0)
    g_ocl = (ga * n_cap).sum(0)
    g_mult = torch.zeros(x.losses.shape[0], dtype=torch.float64, device="cuda")
    for j, elts in enumerate(x.lists):
        on = ((wo[:, j] > 0) & (wo[:, j] < ocl[j])).double()
        cols = []
        for e in elts:
            l = x.losses[int(e)].double()
            f = l * float(x.mult[e]) - float(x.ded[e])
            cols.append(on * l * ((f > 0) & (f < float(x.lim[e]))))
        part = _bags(x, torch.stack(cols, 1))
        g_mult[torch.from_numpy(elts.astype(np.int64)).cuda()] += (part * ga[:, j:j + 1]).sum(0)
    return torch.stack([g_ocr, g_ocl, g_agr, g_agl], 1), g_mult


def exact(case, seed):
    kind, probs = case["kind"], _probs(case)
    if kind == "metrics":
        mean, pml, tvar = _metrics64(_ylt_inputs(case, seed), probs)
        return {"mean": mean, "pml": pml, "tvar": tvar}
    x = _inputs(case, seed)
    ocr, ocl, agr, agl = _cols(x)
    if kind == "payouts":
        occ = _xl(_event_sums64(x, [0]), ocr[:1], ocl[:1])[:, 0]
        T = x.trials
        off = x.trial_off if x.trial_off is not None else torch.arange(T + 1, device="cuda", dtype=torch.int64) * x.k
        pay = torch.empty(x.ids.numel(), dtype=torch.float64, device="cuda")
        ex = torch.empty(T, dtype=torch.int32, device="cuda")
        ylt = torch.empty(T, dtype=torch.float64, device="cuda")
        width = int((off[1:] - off[:-1]).max())
        pos = torch.arange(width, device="cuda")
        step = max(1, (1 << 26) // max(1, width))
        for t0 in range(0, T, step):
            t1 = min(T, t0 + step)
            at = off[t0:t1, None] + pos
            live = at < off[t0 + 1:t1 + 1, None]
            at = at.clamp_(max=x.ids.numel() - 1)
            c = torch.cumsum(torch.where(live, occ[x.ids[at].long()], torch.zeros((), dtype=torch.float64, device="cuda")), 1)
            a = _xl(c, agr[0], agl[0])
            pay[at[live]] = torch.diff(a, dim=1, prepend=torch.zeros_like(a[:, :1]))[live]
            full = live & (c - agr[0] >= agl[0])
            ex[t0:t1] = torch.where(full.any(1), full.int().argmax(1), -1).int()
            ylt[t0:t1] = a[:, -1]
        return {"payouts": pay, "exhaust": ex, "ylt": ylt}
    occ_x = _event_sums64(x)
    s_sum = _bags(x, _xl(occ_x, ocr, ocl))
    ylt = _xl(s_sum, agr, agl).t().contiguous()
    if kind == "price":
        mean, pml, tvar = _metrics64(ylt, probs)
        return {"ylt": ylt, "mean": mean, "pml": pml, "tvar": tvar}
    if kind == "host":
        mean, pml, tvar = _metrics64(ylt, probs)
        return {"mean": mean.cpu(), "pml": pml.cpu(), "tvar": tvar.cpu()}
    if kind == "adjoint":
        w = s_sum - agr
        branch = torch.where(w > agl, 2, ((w > 0) & (w < agl)).int()).to(torch.uint8).t().contiguous()
        terms, mult = _gradients64(x, s_sum, _weights(case, seed), occ_x)
        return {"ylt": ylt, "branch": branch, "terms": terms, "mult": mult}
    if kind == "sensitivity":
        mean, pml, tvar = _metrics64(ylt, probs)
        weights = torch.full_like(ylt, 1.0 / x.trials)
        for q, p in enumerate(probs):
            k = _rank(p, x.trials)
            above, equal = ylt > pml[:, q:q + 1], ylt == pml[:, q:q + 1]
            share = (k - above.sum(1, keepdim=True)) / equal.sum(1, keepdim=True)
            weights += 0.25 / k * (above + equal * share)
        terms, mult = _gradients64(x, s_sum, weights, occ_x)
        return {"mean": mean.cpu(), "tvar": tvar.cpu(), "occ_ret": terms[:, 0].cpu(), "occ_lim": terms[:, 1].cpu(),
                "agg_ret": terms[:, 2].cpu(), "agg_lim": terms[:, 3].cpu(), "mult": mult.cpu()}
    return {"ylt": ylt}
