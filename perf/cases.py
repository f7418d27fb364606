"""The work that users of the search library have it do, as cases that can be
timed: searches of one series (small, large, top-10, wide band, learned
ordering), many queries in one call, queries of ever new lengths, a search of
a series seen for the first time, DTW at given offsets (FP32, extended
precision, without allocations) and the encoder's loss and gradient.

A case is a dict of plain values; ``kind`` says which entry point it calls.
``prepare`` makes the inputs and the handle on the GPU, ``run`` makes one pass
through the public entry points, ``work`` counts what the pass cannot do
without, and ``exact`` gives the outputs in 64 bits by plain torch, sharing no
code with the library (it prunes with its own lower bounds so that long series
stay affordable).  Sizes follow the repository's workloads
(``synth.WORKLOADS``, the benchmark's specs and legs).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1812_10302_gb300 import dtws, train

DEV = "cuda"
NOISE = 0.1  # standard deviation added to a window of the series to make a query


def listed():
    return [
        # the smallest search: a short series already indexed, one short query; launches count
        dict(name="search_1m", kind="search", series="walk", n=1_000_000, m=128, r=6, k=1, ordering="plain"),
        # the flagship search: one query over 1e8 samples, best match
        dict(name="search_100m", kind="search", series="bursts", n=100_000_000, m=512, r=51, k=1, ordering="plain"),
        # top-10 of a medium series at odd sizes (the ten nearest windows, neighbours included)
        dict(name="search_top10", kind="search", series="drift", n=20_000_003, m=999, r=99, k=10, ordering="plain"),
        # the band of nearly the whole query that the paper's experiments sweep up to
        dict(name="search_wide", kind="search", series="bursts", n=20_000_000, m=1024, r=921, k=1, ordering="plain"),
        # a search seeded by the learned proposals
        dict(name="search_learned", kind="search", series="bursts", n=20_000_000, m=1024, r=102, k=1,
             ordering="learned"),
        # a service's batch: queries of uneven length and band in one call, top-10 each
        dict(name="batch", kind="batch", series="walk", n=5_000_000, queries=48, m_lo=128, m_hi=2048, w_lo=0.05,
             w_hi=0.20, k=10),
        # a user who tries one length after another on one series (more lengths than the handle caches)
        dict(name="lengths", kind="lengths", series="walk", n=20_000_000, queries=10, m_lo=128, m_hi=2048, w_lo=0.05,
             w_hi=0.20, k=1),
        # a series seen for the first time: index it, search it once, let it go
        dict(name="cold", kind="cold", series="walk", n=10_000_000, m=512, r=51, k=1),
        # distances of one query to many given windows (labels, features, verification)
        dict(name="dtw_at", kind="dtw_at", series="bursts", n=10_000_000, m=512, r=51, count=100_000),
        # the same in extended precision: a re-score of candidates
        dict(name="rescore", kind="dtw_at_f64", series="walk", n=1_000_000, m=1024, r=102, count=4096),
        # the encoder's training direction: loss and gradient of a held-out set of labelled triples
        dict(name="train_grad", kind="loss_grad", batch=10_000),
        # distances for a host program that owns all device memory (no handle, no allocation)
        dict(name="noalloc", kind="noalloc", series="walk", n=1_000_000, m=256, r=25, count=20_000),
    ]


# ------------------------------------------------------------------ drawn cases
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells(m, r):
    r = min(r, m - 1)
    return m * (2 * r + 1) - r * (r + 1)


def draw(rng):
    kind = rng.choice(["search", "search", "search", "search", "batch", "lengths", "cold", "dtw_at", "dtw_at_f64",
                       "loss_grad", "noalloc"])
    if kind == "loss_grad":
        return dict(kind=kind, batch=_log_int(rng, 64, 10_000))
    series = rng.choice(["walk", "bursts", "drift"])
    if kind == "search":
        ordering = rng.choice(["plain", "plain", "learned"])
        k = rng.choice([1, 1, 3, 10])
        if rng.random() < 0.2:  # a wide band
            m = _log_int(rng, 200, 1500)
            return dict(kind=kind, series=series, n=_log_int(rng, 300_000, 20_000_000), m=m,
                        r=int(rng.uniform(0.5, 0.95) * m), k=1, ordering=ordering)
        m = _log_int(rng, 100, 2048)
        n = _log_int(rng, 300_000, 100_000_000 if k == 1 and m >= 256 else 20_000_000)
        return dict(kind=kind, series=series, n=n, m=m, r=int(rng.uniform(0.03, 0.25) * m), k=k, ordering=ordering)
    if kind in ("batch", "lengths"):
        lo = _log_int(rng, 128, 512)
        return dict(kind=kind, series="walk", n=_log_int(rng, 300_000, 5_000_000 if kind == "batch" else 20_000_000),
                    queries=rng.randint(4, 48) if kind == "batch" else rng.randint(9, 12), m_lo=lo,
                    m_hi=rng.randint(lo + 16, 2048), w_lo=0.05, w_hi=0.20, k=rng.choice([1, 10]) if kind == "batch" else 1)
    if kind == "cold":
        m = _log_int(rng, 100, 2048)
        return dict(kind=kind, series=series, n=_log_int(rng, 300_000, 10_000_000), m=m,
                    r=int(rng.uniform(0.03, 0.25) * m), k=1)
    m = _log_int(rng, 32, 2048)
    w = rng.uniform(0.02, 0.25) if rng.random() < 0.75 else rng.uniform(0.5, 1.0)
    r = min(int(w * m), m - 1)
    most = {"dtw_at": 100_000 * 50_084, "dtw_at_f64": 4096 * 198_186, "noalloc": 20_000 * 12_398}[kind] // _cells(m, r)
    count = min(_log_int(rng, 50, 100_000), max(16, most))
    return dict(kind=kind, series=series, n=_log_int(rng, 300_000, 10_000_000), m=m, r=r, count=count)


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _make_series(kind, n, seed):
    """The three kinds of series of the repository's workloads, FP32 on the GPU: a random walk; a walk with sine
    bursts and N(0, 0.5) noise; a drifting walk whose step variance changes by regimes."""
    g = _generator(seed)
    host = random.Random(int(seed))
    steps = torch.randn(n, generator=g, device=DEV, dtype=torch.float32)
    if kind == "drift":
        s = 0
        while s < n:
            e = min(n, s + int(host.uniform(5e6, 1.5e7)))
            steps[s:e] *= math.sqrt(10.0 ** host.uniform(-1.0, 1.0))
            s = e
        steps += 1e-3
    x = torch.cumsum(steps.double(), 0)
    if kind == "bursts":
        t = host.expovariate(1e-5)
        while t < n:
            s = int(t)
            e = min(n, s + int(host.uniform(1e3, 1e4)))
            per, amp, ph = host.uniform(50.0, 500.0), host.uniform(1.0, 5.0), host.uniform(0.0, 2 * math.pi)
            x[s:e] += amp * torch.sin(torch.arange(e - s, device=DEV, dtype=torch.float64) * (2 * math.pi / per) + ph)
            t += host.expovariate(1e-5)
        x += 0.5 * torch.randn(n, generator=g, device=DEV, dtype=torch.float32)
    return x.float()


def _queries(case, x, seed):
    """(queries, r, true offsets): noisy copies of windows at uniform offsets."""
    host = random.Random(int(seed) * 7919 + 1)
    g = _generator(seed * 31 + 5)
    if case["kind"] in ("batch", "lengths"):
        sizes = []
        for i in range(case["queries"]):
            m = host.randint(case["m_lo"], case["m_hi"])
            while case["kind"] == "lengths" and any(m == t[0] for t in sizes):
                m = host.randint(case["m_lo"], case["m_hi"])
            sizes.append((m, int(host.uniform(case["w_lo"], case["w_hi"]) * m)))
    else:
        sizes = [(case["m"], case["r"])]
    qs, rs, at = [], [], []
    for m, r in sizes:
        o = host.randrange(x.numel() - m + 1)
        qs.append(x[o:o + m] + NOISE * torch.randn(m, generator=g, device=DEV, dtype=torch.float32))
        rs.append(r)
        at.append(o)
    return qs, rs, at


def _offsets(case, at, seed):
    """Offsets of the windows to score: uniform ones, and the query's own neighbourhood among them."""
    N = case["n"] - case["m"] + 1
    o = torch.randint(0, N, (case["count"],), generator=_generator(seed * 131 + 3), device=DEV, dtype=torch.int64)
    near = min(8, case["count"])
    o[:near] = torch.clamp(torch.arange(near, device=DEV) + at, max=N - 1)
    return o


def _triples(case, seed):
    """(params, uq, uc, y): the committed parameters and encoder inputs as the training data has them -- half the
    candidates near their query's window, half anywhere -- with labels of the size of DTW / m."""
    B, m, n = case["batch"], 1024, 2_000_000
    x = _make_series("bursts", n, seed)
    xq = x + NOISE * torch.randn(n, generator=_generator(seed + 17), device=DEV, dtype=torch.float32)
    rng = np.random.default_rng(seed)
    q = rng.integers(0, n - m + 1, B)
    c = np.where(rng.random(B) < 0.5, np.clip(q + rng.integers(-m // 8, m // 8 + 1, B), 0, n - m),
                 rng.integers(0, n - m + 1, B))
    near = np.abs(q - c) <= m // 8
    y = np.where(near, 10.0 ** rng.uniform(-3.0, -0.5, B), rng.uniform(0.05, 1.0, B)).astype(np.float32)
    uq, uc = dtws.enc_prep(xq, q, m), dtws.enc_prep(x, c, m)
    return train.load_weights(), uq, uc, y


def prepare(case, seed):
    kind = case["kind"]
    if kind == "loss_grad":
        return dict(case=case, args=[torch.from_numpy(a).to(DEV) for a in _triples(case, seed)])
    x = _make_series(case["series"], case["n"], seed)
    qs, rs, at = _queries(case, x, seed)
    st = dict(case=case, q=qs[0], r=rs[0])
    if kind == "cold":
        st["x"] = x
        return st
    if kind == "noalloc":
        st.update(x=x, offsets=_offsets(case, at[0], seed),
                  out=torch.empty(case["count"], dtype=torch.float32, device=DEV))
        return st
    st["ix"] = dtws.Index(x)
    if kind == "search":
        if case["ordering"] == "learned":
            st["ix"].set_encoder(train.load_weights())
            st["ix"].set_options(ordering=dtws.DTWS_ORDER_LEARNED)
        st["out"] = (torch.empty(case["k"], dtype=torch.int64, device=DEV),
                     torch.empty(case["k"], dtype=torch.float32, device=DEV))
    elif kind in ("batch", "lengths"):
        st["qs"] = [q.cpu().numpy() for q in qs]
        st["rs"] = rs
    else:
        st["offsets"] = _offsets(case, at[0], seed)
    return st


# ------------------------------------------------------------------ one pass
def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "search":
        return state["ix"].query(state["q"], state["r"], case["k"], out=state["out"])
    if kind == "batch":
        return state["ix"].query_batch(state["qs"], state["rs"], case["k"])
    if kind == "lengths":
        got = [state["ix"].query(q, r, case["k"]) for q, r in zip(state["qs"], state["rs"])]
        return np.stack([i for i, _ in got]), np.stack([d for _, d in got])
    if kind == "cold":
        with dtws.Index(state["x"]) as ix:
            return ix.query(state["q"], state["r"], case["k"])
    if kind == "dtw_at":
        return state["ix"].dtw_at(state["q"], state["r"], state["offsets"])
    if kind == "dtw_at_f64":
        return state["ix"].dtw_at_f64(state["q"], state["r"], state["offsets"])
    if kind == "loss_grad":
        return dtws.enc_loss_grad(*state["args"])
    x, q, o, out = state["x"], state["q"], state["offsets"], state["out"]
    status = dtws.load().dtws_dtw_at_noalloc(x.data_ptr(), x.numel(), q.data_ptr(), q.numel(), state["r"],
                                             o.data_ptr(), o.numel(), out.data_ptr(),
                                             torch.cuda.current_stream().cuda_stream)
    if status != dtws.DTWS_OK:
        raise dtws.DtwsError(status, "dtws_dtw_at_noalloc")
    return out


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "loss_grad":
        # 2 sequences per triple; the four convolutions and the projection, forward, data and weight gradients
        macs = 57 * 32 * 7 + (51 + 45 + 39) * 32 * 32 * 7 + 64 * 256
        B = case["batch"]
        return dict(bytes=2 * B * 64 * 4 + B * 4 + 2 * 38112 * 4, flops=2 * B * 3 * 2 * macs)
    n = case["n"]
    if kind in ("search", "cold"):
        # every sample once; per window the normalised end points and their squared distances (Eq. 7)
        return dict(bytes=4 * n + 4 * case["m"] + 12 * case["k"], flops=10 * (n - case["m"] + 1))
    if kind in ("batch", "lengths"):
        # the series once per call of the library; every window of every query bounded
        calls = 1 if kind == "batch" else case["queries"]
        m = (case["m_lo"] + case["m_hi"]) // 2
        return dict(bytes=4 * n * calls + case["queries"] * (4 * m + 12 * case["k"]), flops=10 * n * case["queries"])
    # DTW at offsets: subtract, multiply-add, two minima per band cell; the samples the windows cover
    size = 8 if kind == "dtw_at_f64" else 4
    return dict(bytes=4 * min(n, case["count"] * case["m"]) + case["count"] * (8 + size) + 4 * case["m"],
                flops=5 * case["count"] * _cells(case["m"], case["r"]))


# ------------------------------------------------------------------ the outputs in 64 bits
_INF = float("inf")


def _normalise(w):
    """z-normalisation of rows (population deviation; variance <= 1e-24 max(1, mean^2): all zeros)."""
    mu = w.mean(1, keepdim=True)
    d = w - mu
    var = d.square().mean(1, keepdim=True)
    zero = var <= 1e-24 * torch.clamp(mu.square(), min=1.0)
    return torch.where(zero, torch.zeros_like(d), d / torch.sqrt(torch.where(zero, torch.ones_like(var), var)))


def _windows(x, offsets, m):
    return _normalise(x[offsets[:, None] + torch.arange(m, device=DEV)].double())


def _dtw(qh, W, r):
    """Banded DTW of the query to every row of W along anti-diagonals, all rows at once; D[i] is cell (i, a - i)."""
    m, B = qh.numel(), W.shape[0]
    C = W.t().contiguous()
    prev = torch.full((m + 1, B), _INF, device=DEV, dtype=torch.float64)  # row i + 1 holds index i
    prev2, cur = prev.clone(), prev.clone()
    prev2[0] = 0.0  # the cell (-1, -1)
    rev = torch.arange(m - 1, -1, -1, device=DEV)
    Crev = C[rev]  # row u: sample m - 1 - u
    for a in range(2 * m - 1):
        lo, hi = max(0, a - m + 1, (a - r + 1) // 2), min(a, m - 1, (a + r) // 2)
        cur.fill_(_INF)
        if lo <= hi:
            j0 = m - 1 - (a - lo)  # row of Crev for cell lo
            cost = (qh[lo:hi + 1, None] - Crev[j0:j0 + hi - lo + 1]).square_()
            best = torch.minimum(torch.minimum(prev[lo:hi + 1], prev[lo + 1:hi + 2]), prev2[lo:hi + 1])
            cur[lo + 1:hi + 2] = cost + best
        prev2, prev, cur = prev, cur, prev2
    return prev[m].clone()


def _dtw_at(x, q, r, offsets, block=None):
    qh = _normalise(q.double()[None])[0]
    m = qh.numel()
    block = block or max(256, min(16384, int(3e8 // m)))
    return torch.cat([_dtw(qh, _windows(x, o, m), min(r, m - 1)) for o in offsets.split(block)])


def _search(x, q, r, k, near, most=3_000_000):
    """(offsets, distances) of the k best windows, or None when more than ``most`` windows stay after LB_KimFL: the
    end-point bound for every window, then LB_Keogh against the query's envelope, then DTW from the smallest bound
    on, against the k-th best found so far (from the windows around ``near``)."""
    m, N = q.numel(), x.numel() - q.numel() + 1
    r = min(r, m - 1)
    qh = _normalise(q.double()[None])[0]
    first = torch.arange(max(0, near - 2 * k), min(N, near + 2 * k + 1), device=DEV)
    found = [(first, _dtw_at(x, q, r, first))]
    thr = float(found[0][1].sort().values[k - 1])
    chunk, keep = 1 << 22, []
    for c0 in range(0, N, chunk):
        c1 = min(N, c0 + chunk)
        xs = x[c0:c1 + m - 1].double()
        xs -= xs[0].clone()
        s1 = torch.cumsum(torch.nn.functional.pad(xs, (1, 0)), 0)
        s2 = torch.cumsum(torch.nn.functional.pad(xs.square(), (1, 0)), 0)
        mu = (s1[m:] - s1[:-m]) / m
        sg = torch.sqrt(torch.clamp((s2[m:] - s2[:-m]) / m - mu.square(), min=1e-30))
        kim = ((xs[:c1 - c0] - mu) / sg - qh[0]).square() + ((xs[m - 1:] - mu) / sg - qh[-1]).square()
        keep.append(torch.nonzero(kim <= thr * (1 + 1e-4) + 1e-5)[:, 0] + c0)
    keep = torch.cat(keep)
    if keep.numel() > most:
        return None
    up = torch.nn.functional.max_pool1d(qh[None, None], 2 * r + 1, 1, r)[0, 0]
    dn = -torch.nn.functional.max_pool1d(-qh[None, None], 2 * r + 1, 1, r)[0, 0]
    lb = []
    for o in keep.split(max(256, int(2e8 // m))):
        W = _windows(x, o, m)
        lb.append((torch.clamp(W - up, min=0.0) + torch.clamp(dn - W, min=0.0)).square_().sum(1))
    lb, order = torch.cat(lb).sort()
    keep = keep[order]
    block = max(256, min(8192, int(1e8 // m)))
    for s in range(0, keep.numel(), block):
        if float(lb[s]) > thr * (1 + 1e-9):
            break
        o = keep[s:s + block][lb[s:s + block] <= thr * (1 + 1e-9)]
        found.append((o, _dtw_at(x, q, r, o)))
        d = torch.cat([f[1] for f in found])
        i = torch.cat([f[0] for f in found])
        i, u = np.unique(i.cpu().numpy(), return_index=True)
        d = d.cpu().numpy()[u]
        best = np.lexsort((i, d))[:max(4 * k, 16)]
        found = [(torch.from_numpy(i[best]).to(DEV), torch.from_numpy(d[best]).to(DEV))]
        thr = float(np.sort(d)[k - 1])
    i, d = found[0][0].cpu().numpy(), found[0][1].cpu().numpy()
    best = np.lexsort((i, d))[:k]
    return i[best], d[best]


def _loss_grad(params, uq, uc, y):
    """The encoder's training loss and its gradient by autograd."""
    p = params.double().clone().requires_grad_(True)
    sizes = [32 * 7, 32 * 7 * 32, 32 * 7 * 32, 32 * 7 * 32, 64 * 256]
    w1, w2, w3, w4, proj = p.split(sizes)
    convs = [w1.view(32, 7, 1)] + [w.view(32, 7, 32) for w in (w2, w3, w4)]

    def embed(u):
        h = u[:, None, :63].double()
        for i, w in enumerate(convs):
            h = torch.nn.functional.conv1d(h, w.transpose(1, 2))
            h = torch.relu(h) if i < 3 else h
        cut = [39 * s // 8 for s in range(9)]
        pooled = torch.stack([h[:, :, cut[s]:cut[s + 1]].mean(2) for s in range(8)], 1)
        return pooled.reshape(u.shape[0], 256) @ proj.view(64, 256).t()

    dist = (embed(uq) - embed(uc)).square().sum(1)
    loss = (torch.log(dist + 1e-3) - torch.log(y.double() + 1e-3)).square().mean()
    loss.backward()
    return float(loss), p.grad.detach()


def exact(case, seed):
    kind = case["kind"]
    if kind == "loss_grad":
        return _loss_grad(*[torch.from_numpy(a).to(DEV) for a in _triples(case, seed)])
    if kind in ("batch", "lengths") and case["n"] * case["queries"] > 2e7:
        return None  # minutes
    x = _make_series(case["series"], case["n"], seed)
    qs, rs, at = _queries(case, x, seed)
    if kind in ("dtw_at", "dtw_at_f64", "noalloc"):
        return _dtw_at(x, qs[0], rs[0], _offsets(case, at[0], seed))
    got = [_search(x, q, r, case["k"], o, 3_000_000 // len(qs)) for q, r, o in zip(qs, rs, at)]
    if any(g is None for g in got):
        return None
    if kind in ("search", "cold"):
        return list(got[0])
    return [np.stack([g[0] for g in got]), np.stack([g[1] for g in got])]
