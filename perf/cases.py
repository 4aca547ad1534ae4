"""The calls whose time matters to a user of the library, over the sizes it is used at.

Inputs are the synthetic matrix-factorisation-like vectors of the repository's workloads
(Gaussian directions, log-normal norms: sigma 0.3 for users, 0.5 for items), drawn on the
GPU.  With ``grid`` every row is rounded to the 2^-12 grid of its own power of two (exact
scores are then integer sums); without it the rows are the plain FP32 vectors
that a trainer writes (exact scores are FP64 sums).  ``plain`` cases are i.i.d. N(0, 0.25)
entries.  The paper's own vectors have d = 200.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2504_13445_gb300 as rkm

CATALOGUE_ITEMS = 300_000  # items the resident users' thresholds come from (serving workload)


def listed():
    return [
        # Small interactive call: one shop's users and items, the latency of a whole top-N.
        dict(name="topn_2k", kind="topn", n=2_000, m=1_000, d=32, k=10, N=10, plain=True, grid=True,
             precision="bf16"),
        # A mid-size problem on the plain FP32 path (no reduced-precision operands).
        dict(name="topn_20k_fp32", kind="topn", n=20_000, m=5_000, d=64, k=25, N=50, plain=False, grid=True,
             precision="fp32"),
        # The FP8 operand option on an ordinary catalogue.
        dict(name="topn_100k_fp8", kind="topn", n=100_000, m=50_000, d=128, k=10, N=100, plain=False, grid=True,
             precision="fp8"),
        # Ordinary nightly job on quantised vectors.
        dict(name="topn_500k", kind="topn", n=500_000, m=100_000, d=64, k=25, N=50, plain=False, grid=True,
             precision="bf16"),
        # The largest single-GPU problem of the benchmark.
        dict(name="topn_2m", kind="topn", n=2_000_000, m=500_000, d=128, k=10, N=100, plain=False, grid=True,
             precision="bf16"),
        # Many users, short catalogue, deep trained FP32 vectors (the paper's d = 200, N = 20).
        dict(name="topn_480k_d200", kind="topn", n=480_189, m=17_770, d=200, k=10, N=20, plain=False, grid=False,
             precision="bf16"),
        # Offline half of the offline/online split: lists S_kmax(u) at the largest k used, odd sizes.
        dict(name="thresholds_130k_k50", kind="thresholds", n=130_051, m=30_011, d=100, k=50, plain=False,
             grid=False, precision="bf16"),
        # Scores of a whole catalogue against stored thresholds (no filter: every item is wanted).
        dict(name="scores_100k", kind="scores", n=100_000, m=40_000, d=64, k=20, plain=False, grid=True,
             precision="bf16"),
        # A few what-if items against a million resident users: the latency of a single query.
        dict(name="query_32", kind="query", n=1_000_000, m=CATALOGUE_ITEMS, d=100, k=20, q=32, plain=False,
             grid=True, precision="bf16"),
        # A burst of what-if requests through the serving loop, sizes log-uniform in [1, 4096].
        dict(name="serve_64", kind="serve", n=1_000_000, m=CATALOGUE_ITEMS, d=100, k=20, requests=64, plain=False,
             grid=True, precision="bf16"),
        # Many tenants in one call: uneven instances of one batch.
        dict(name="batch_16", kind="batch", count=16, n_lo=10_000, n_hi=200_000, m_lo=5_000, m_hi=50_000, k=10,
             N=20, plain=False, grid=True, precision="bf16"),
        # End to end from host memory: the copies are part of the call.
        dict(name="host_200k", kind="host", n=200_000, m=50_000, d=96, k=20, N=50, plain=False, grid=False,
             precision="bf16"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["topn", "topn", "topn", "thresholds", "scores", "query", "query", "serve", "batch", "host"])
    precision = rng.choice(["bf16"] * 6 + ["fp8", "fp32"]) if kind in ("topn", "thresholds", "scores") else "bf16"
    grid = rng.random() < 0.5
    if kind in ("query", "serve"):
        c = dict(kind=kind, n=_log(rng, 50_000, 1_000_000), m=_log(rng, 10_000, CATALOGUE_ITEMS),
                 d=rng.randint(32, 200), k=rng.choice([5, 10, 20, 25]))
        if kind == "query":
            c["q"] = _log(rng, 32, 4096)
        else:
            c["requests"] = rng.randint(16, 64)
    elif kind == "batch":
        c = dict(kind=kind, count=rng.randint(3, 16), n_lo=_log(rng, 1_000, 20_000), n_hi=_log(rng, 30_000, 200_000),
                 m_lo=_log(rng, 500, 10_000), m_hi=_log(rng, 15_000, 50_000), k=rng.choice([5, 10, 25]), N=20)
    else:
        big = precision == "bf16" and kind != "host"
        n = _log(rng, 1_500, 700_000 if big else 200_000 if kind == "host" else 50_000)
        m = _log(rng, 700, 150_000 if big else 50_000 if kind == "host" else 20_000)
        c = dict(kind=kind, n=n, m=m, d=rng.choice([rng.randint(8, 64), rng.randint(65, 128), rng.randint(129, 256)]),
                 k=rng.choice([1, 5, 10, 20, 25, 50]))
        if kind in ("topn", "host"):
            c["N"] = rng.choice([1, 10, 20, 50, 100, 500])
    return dict(c, plain=False, grid=grid, precision=precision)


# ---------------------------------------------------------------- inputs

def _quantise(x):
    """Round each row to the grid 2^(e - 12), e the smallest integer with max|x| <= 2^e."""
    f, e = torch.frexp(x.abs().amax(dim=1, keepdim=True))
    e = torch.where(f == 0.5, e - 1, e).to(torch.int32)
    up = ((12 - e + 127) << 23).view(torch.float32)  # 2^(12 - e), exactly
    down = ((e - 12 + 127) << 23).view(torch.float32)
    return torch.round(x * up) * down


def _rows(case, count, d, sigma, gen):
    x = torch.randn(count, d, device="cuda", dtype=torch.float32, generator=gen)
    if case["plain"]:
        x = (x * 0.5).clamp_(-1.0, 1.0)
        return torch.round(x * 4096.0) / 4096.0 if case["grid"] else x
    norm = torch.exp(sigma * torch.randn(count, 1, device="cuda", dtype=torch.float32, generator=gen))
    x = x * (norm / x.norm(dim=1, keepdim=True))
    return _quantise(x) if case["grid"] else x


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 31))


def _users_items(case, seed):
    g = _gen(seed)
    return _rows(case, case["n"], case["d"], 0.3, g), _rows(case, case["m"], case["d"], 0.5, g)


def _sizes(case, seed):
    """Batch: the instances' (n, m, d, N), log-uniform; the depths in turn."""
    r = np.random.default_rng(case["count"] * 7919 + case["n_lo"])  # the layout belongs to the case
    out = []
    for j in range(case["count"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        m = int(round(math.exp(r.uniform(math.log(case["m_lo"]), math.log(case["m_hi"])))))
        out.append((n, m, (32, 64, 128)[j % 3], min(case["N"], m)))
    return out


def _request_sizes(case):
    """Serving: request sizes log-uniform in [1, 4096]."""
    r = np.random.default_rng(case["requests"])
    return [int(min(4096, max(1, math.floor(math.exp(x * math.log(4097.0)))))) for x in r.random(case["requests"])]


def _n_out(case):
    return min(case["N"], case["m"])


def _k(case):
    return min(case["k"], case["m"])


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case, ctx=rkm.Context(case["precision"]))
    if kind == "batch":
        g = _gen(seed)
        s["problems"] = [(_rows(case, n, d, 0.3, g), _rows(case, m, d, 0.5, g), case["k"], N)
                         for n, m, d, N in _sizes(case, seed)]
        s["outs"] = [(torch.empty(N, dtype=torch.int32, device="cuda"), torch.empty(N, dtype=torch.int32, device="cuda"))
                     for *_, N in s["problems"]]
        return s
    U, P = _users_items(case, seed)
    if kind in ("query", "serve"):
        # Thresholds of the resident users against the catalogue, in a context of its own
        # whose workspace is given back.
        with rkm.Context(case["precision"]) as c:
            tau, tid, _ = c.thresholds(U, P, _k(case))
        s["ctx"].resident_set(U, tau, tid)
        g = _gen(seed + 77)
        if kind == "query":
            s["Q"] = _rows(case, case["q"], case["d"], 0.5, g)
        else:
            sizes = _request_sizes(case)
            rows = _rows(case, sum(sizes), case["d"], 0.5, g).cpu().numpy()
            cuts = np.cumsum([0] + sizes)
            s["requests"] = [np.ascontiguousarray(rows[a:b]) for a, b in zip(cuts[:-1], cuts[1:])]
            s["server"] = rkm.Server(s["ctx"], memory_bytes=256 << 20)
        return s
    if kind == "host":
        s["U"], s["P"] = (x.cpu().pin_memory().numpy() for x in (U, P))
        return s
    s["U"], s["P"] = U, P
    if kind == "scores":
        with rkm.Context(case["precision"]) as c:
            s["tau"], s["tid"], _ = c.thresholds(U, P, _k(case))
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "topn":
        return ctx.topn(s["U"], s["P"], _k(case), _n_out(case), return_thresholds=True)
    if kind == "thresholds":
        return ctx.thresholds(s["U"], s["P"], _k(case), want_topk=True)
    if kind == "scores":
        return ctx.scores(s["U"], s["P"], s["tau"], s["tid"])
    if kind == "query":
        return ctx.query_new_items(s["Q"])
    if kind == "serve":
        srv = s["server"]
        tickets = [srv.submit(q) for q in s["requests"]]
        return np.concatenate([srv.wait(t)[0] for t in tickets])
    if kind == "batch":
        return [x for pair in ctx.topn_batch(s["problems"], s["outs"]) for x in pair]
    return ctx.topn_host(s["U"], s["P"], _k(case), _n_out(case))


def work(case):
    """Inputs read once, outputs written once; 2 d n m operations for one dense product of
    users and items (the Cauchy-Schwarz bounds let a call skip some of the pairs)."""
    kind = case["kind"]
    if kind == "batch":
        sz = _sizes(case, 0)
        return dict(bytes=sum(4.0 * d * (n + m) + 8 * N for n, m, d, N in sz),
                    flops=sum(2.0 * d * n * m for n, m, d, N in sz))
    n, d = case["n"], case["d"]
    m = case["m"] if kind not in ("query", "serve") else case["q"] if kind == "query" else sum(_request_sizes(case))
    out = {"topn": 12 * n, "thresholds": (12 + 4 * case["k"]) * n, "scores": 12 * n + 4 * m, "query": 12 * n + 4 * m,
           "serve": 12 * n + 4 * m, "host": 0}[kind]
    return dict(bytes=4.0 * d * (n + m) + out + 8 * case.get("N", 0), flops=2.0 * d * n * m)


def exact(case, seed):
    """tau_u in FP64 (the k-th largest inner product), where it is an output and quick enough."""
    if case["kind"] not in ("topn", "thresholds") or float(case["n"]) * case["m"] * (case["d"] + 128) > 1.2e13:
        return None
    U, P = _users_items(case, seed)
    P64 = P.double().t().contiguous()
    k = _k(case)
    step = max(1, (1 << 28) // case["m"])
    tau = torch.cat([torch.topk(U[a:a + step].double() @ P64, k, dim=1, sorted=True).values[:, k - 1]
                     for a in range(0, case["n"], step)]) + 0.0
    return (None, None, tau, None) if case["kind"] == "topn" else (tau, None, None)
