"""What this library is asked to do, as cases that can be timed.

Each case is one call (or the one replay) that a user's program makes through the package's public
binding, on synthetic rows of the shapes the library's own workloads have: integer rows 0..255 (the
SIFT-shaped Gaussian mixture and the tiny one), floats in [0, 1] (GIST-shaped) and unit vectors
(DEEP-shaped).  Rows are drawn on the GPU from the case's seed; a search's index is built by
``prepare`` (a program builds it once and keeps it).

Calls:
  search  Index.search: FP32 search of a device batch
  ex      Index.search_ex: the precision forms (BF16 / FP8 / 8-bit copies, FP32 re-rank when lossy)
  host    Index.search_host: the same on page-locked host buffers, copies included
  plan    Index.plan(...).run(): uneven k and L, autotuned, replayed as a CUDA graph
  oneshot Index.search_batched: uneven k and L without a plan
  truth   nsg_knn_query: exact k nearest rows of a query batch (ground truth)
  graph   nsg_knn_init: the exact kNN graph the build starts from
  build   nsg_build: the whole index construction on the exact kNN graph
  descent nsg_build_ex: the same on a kNN graph by nn-descent
"""
import math

import torch

from paper_1707_00143_gb300 import capi

PREC = {"f32": capi.PREC_F32, "bf16": capi.PREC_BF16, "fp8": capi.PREC_FP8, "u8": capi.PREC_U8}
ROW_BYTES = {"f32": 4, "bf16": 2, "fp8": 1, "u8": 1}

# build parameters by kind of rows: kNN degree, pool, degree bound, candidate cap, kNN by nn-descent
BUILD = {
    "tiny": dict(K=20, L=40, R=16, C=200),
    "sift": dict(K=100, L=40, R=50, C=500),
    "gist": dict(K=100, L=60, R=70, C=500),
    "deep": dict(K=64, L=60, R=32, C=500),
}
COMPONENTS = {"tiny": 16, "sift": 100, "gist": 50, "deep": 1000}
DESCENT = (16, 16, 12, 0.001, 1)  # samples, reverse samples, iterations, stopping share, seed


def listed():
    return [
        # a single interactive query: the latency of one search
        dict(name="search_one", call="search", data="sift", n=100_000, d=128, nq=1, k=10, L=100, prec="f32"),
        # the SIFT-shaped batch in the plain FP32 form
        dict(name="search_sift_f32", call="search", data="sift", n=300_000, d=128, nq=10_000, k=100, L=150, prec="f32"),
        # the SIFT-shaped batch at full size in the exact 8-bit form: the headline operating point
        dict(name="search_sift_u8", call="ex", data="sift", n=1_000_000, d=128, nq=10_000, k=100, L=138, prec="u8"),
        # wide float rows through the BF16 copy with the FP32 re-rank, 1,000 queries
        dict(name="search_gist_bf16", call="ex", data="gist", n=100_000, d=960, nq=1_000, k=100, L=300, prec="bf16"),
        # a serving call on host buffers: a ragged batch of rows whose width is no power of two, FP8 copy
        dict(name="search_host_fp8", call="host", data="gist", n=60_000, d=100, nq=777, k=10, L=120, prec="fp8"),
        # uneven queries (k of 1, 10, 100, L of 20 to 500) in one replayed launch, lossy 8-bit copy
        dict(name="plan_deep_u8", call="plan", data="deep", n=300_000, d=96, nq=20_000, k=100, L=500, prec="u8"),
        # ground truth of a small batch on a small base: mostly launches
        dict(name="truth_tiny", call="truth", data="tiny", n=10_000, d=32, nq=100, k=10),
        # ground truth of the GIST-shaped batch at full size: wide float rows, few queries
        dict(name="truth_gist", call="truth", data="gist", n=1_000_000, d=960, nq=1_000, k=100),
        # the exact kNN graph of integer rows, ragged size
        dict(name="graph_sift", call="graph", data="sift", n=300_007, d=128, k=100),
        # a small index, whole construction
        dict(name="build_tiny", call="build", data="tiny", n=10_000, d=32),
        # the SIFT-shaped construction at a tenth of its size
        dict(name="build_sift", call="build", data="sift", n=100_000, d=128),
        # the DEEP-shaped construction on an nn-descent graph
        dict(name="build_deep", call="descent", data="deep", n=150_000, d=96),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call = rng.choice(["search", "search", "ex", "ex", "ex", "host", "plan", "oneshot", "truth", "truth", "graph",
                       "build", "descent"])
    data = "deep" if call == "descent" else rng.choice(["tiny", "sift", "gist", "deep"])
    d = {"tiny": lambda: rng.randint(17, 64), "sift": lambda: rng.randint(65, 160),
         "gist": lambda: _log(rng, 48, 960), "deep": lambda: rng.randint(48, 200)}[data]()
    if call == "truth":
        n, nq = _log(rng, 5_000, 500_000), _log(rng, 1, 10_000)
        nq = max(1, min(nq, int(9e11 / (n * d))))
        return dict(call=call, data=data, n=n, d=d, nq=nq, k=rng.choice([1, 10, 100]))
    if call == "graph":
        return dict(call=call, data=data, n=_log(rng, 5_000, 200_000), d=min(d, 160), k=rng.choice([20, 64, 100]))
    if call in ("build", "descent"):
        return dict(call=call, data=data, n=_log(rng, 5_000, 60_000 if d <= 200 else 20_000), d=d)
    n = _log(rng, 10_000, 200_000 if d <= 200 else 40_000)
    L = _log(rng, 20, 1_200)
    nq = _log(rng, 1, min(10_000, max(64, int(2e8 / (L * d)))))
    k = min(rng.choice([1, 10, 100]), L)
    prec = "f32" if call == "search" else rng.choice(["f32", "bf16", "fp8", "u8", "u8"])
    if call in ("plan", "oneshot"):
        k, L = 100, max(L, 100)
    return dict(call=call, data=data, n=n, d=d, nq=nq, k=k, L=L, prec=prec)


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + stream) % (1 << 62))
    return g


def _rows(data, n, d, seed, stream):
    """n rows of the mixture that `seed` gives; streams 1 (base) and 2 (queries) share its centres."""
    gc, g = _generator(seed, 0), _generator(seed, stream)
    m = COMPONENTS[data]
    comp = torch.randint(0, m, (n,), generator=g, device="cuda")
    if data == "deep":
        cen = torch.randn((m, d), generator=gc, device="cuda")
        cen /= cen.norm(dim=1, keepdim=True)
        sigma = 0.05
    elif data == "gist":
        cen = torch.rand((m, d), generator=gc, device="cuda") * 0.6 + 0.2
        sigma = 0.1
    else:
        cen = torch.rand((m, d), generator=gc, device="cuda") * 175.0 + 40.0
        sigma = 30.0
    x = torch.randn((n, d), generator=g, device="cuda").mul_(sigma)
    for a in range(0, n, 1 << 18):
        x[a:a + (1 << 18)] += cen[comp[a:a + (1 << 18)]]
    if data == "deep":
        x /= x.norm(dim=1, keepdim=True)
    elif data == "gist":
        x.clamp_(0.0, 1.0)
    else:
        x.round_().clamp_(0.0, 255.0)
    return x


def _build(data, base, descent):
    b = BUILD[data]
    knn = capi.NnDescentParams(*DESCENT) if descent else None
    return capi.nsg_build_ex(base, b["K"], b["L"], b["R"], b["C"], seed=0, knn_params=knn)


def prepare(case, seed):
    call, data, n, d = case["call"], case["data"], case["n"], case["d"]
    base = _rows(data, n, d, seed, 1)
    if call in ("graph", "build", "descent"):
        return dict(case=case, base=base)
    q = _rows(data, case["nq"], d, seed, 2)
    if call == "truth":
        return dict(case=case, base=base, q=q)
    index = _build(data, base, data == "deep")
    prec = PREC[case["prec"]]
    if prec:
        index.prepare(prec)
    s = dict(case=case, index=index, q=q, params=capi.SearchParams(precision=prec))
    if call == "host":
        nq, k = case["nq"], case["k"]
        s["q"] = q.cpu().pin_memory()
        s["ids"] = torch.empty((nq, k), dtype=torch.int32).pin_memory()
        s["d2"] = torch.empty((nq, k), dtype=torch.float32).pin_memory()
    if call in ("plan", "oneshot"):
        g = _generator(seed, 3)
        ks = torch.tensor([1, 10, 100], dtype=torch.int32, device="cuda")
        k = ks[torch.randint(0, 3, (case["nq"],), generator=g, device="cuda")].contiguous()
        L = torch.randint(20, case["L"] + 1, (case["nq"],), generator=g, device="cuda", dtype=torch.int32)
        s["k"], s["L"] = k, torch.maximum(L, k)
        if call == "plan":
            s["plan"] = index.plan(q, s["k"], s["L"], kmax=case["k"], Lmax=case["L"], params=s["params"])
    return s


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "search":
        ids, d2 = state["index"].search(state["q"], case["k"], case["L"])
    elif call == "ex":
        out = state["index"].search_ex(state["q"], case["k"], case["L"], params=state["params"], counters=False)
        ids, d2 = out["ids"], out["d2"]
    elif call == "host":
        out = state["index"].search_host(state["q"], case["k"], case["L"], params=state["params"], ids=state["ids"],
                                         d2=state["d2"])
        ids, d2 = out["ids"], out["d2"]
    elif call == "plan":
        ids, d2 = state["plan"].run()
    elif call == "oneshot":
        out = state["index"].search_batched(state["q"], state["k"], state["L"], kmax=case["k"], Lmax=case["L"],
                                            params=state["params"])
        ids, d2 = out["ids"], out["d2"]
    elif call == "truth":
        ids, d2 = capi.nsg_knn_query(state["base"], state["q"], case["k"])
    elif call == "graph":
        ids, d2 = capi.nsg_knn_init(state["base"], case["k"])
    else:
        index = _build(case["data"], state["base"], call == "descent")
        adj, deg = index.graph()
        return dict(adj=adj, deg=deg, nav=index.info()["nav"])
    return dict(ids=ids, d2=d2)


def work(case):
    """Inputs read once, outputs written once, and the distances the method measures (a search checks
    about L nodes and measures about half of each one's neighbours)."""
    call, n, d = case["call"], case["n"], case["d"]
    b = BUILD[case["data"]]
    if call == "truth":
        return dict(bytes=4.0 * d * (n + case["nq"]) + 8.0 * case["nq"] * case["k"], flops=2.0 * case["nq"] * n * d)
    if call == "graph":
        return dict(bytes=4.0 * d * n + 8.0 * n * case["k"], flops=2.0 * n * n * d)
    if call in ("build", "descent"):
        knn = 2.0 * n * n * d if call == "build" else DESCENT[2] * n * 500.0 * 3 * d
        collect = n * 0.5 * b["K"] * b["L"] * 3.0 * d
        prune = n * b["R"] * b["R"] * 3.0 * d
        return dict(bytes=4.0 * d * n + 4.0 * n * (b["R"] + 1), flops=knn + collect + prune)
    nq, L = case["nq"], case["L"]
    if call in ("plan", "oneshot"):
        L = 0.5 * (L + 20)
    row = ROW_BYTES[case["prec"]] * d
    gather = nq * (L * b["R"] * 4.0 + 0.5 * L * b["R"] * row)
    index = n * (row + 4.0 * b["R"])
    return dict(bytes=min(gather, index) + 4.0 * nq * d + 8.0 * nq * case["k"], flops=nq * 0.5 * L * b["R"] * 3.0 * d)


def exact(case, seed):
    """Distances of the k nearest rows in 64 bits for the exact calls.  A graph search's results follow
    the index it walks, so it has no value that is independent of this library."""
    if case["call"] not in ("truth", "graph"):
        return None
    n, d, k = case["n"], case["d"], case["k"]
    join = case["call"] == "graph"
    nq = n if join else case["nq"]
    if 2.0 * nq * n * d > 5e12 or nq * n > 4e9:
        return None
    base = _rows(case["data"], n, d, seed, 1)
    q = base if join else _rows(case["data"], nq, d, seed, 2)
    out = []
    for a in range(0, nq, 1024):
        qd = q[a:a + 1024].double()
        best = None
        for c in range(0, n, 1 << 17):
            x = base[c:c + (1 << 17)].double()
            d2 = (x * x).sum(1) + (qd * qd).sum(1, keepdim=True) - 2.0 * (qd @ x.T)
            if join:
                r = torch.arange(a, a + len(qd), device="cuda")
                inside = (r >= c) & (r < c + len(x))
                d2[inside.nonzero()[:, 0], r[inside] - c] = math.inf
            v = torch.topk(d2, min(k, len(x)), dim=1, largest=False).values
            best = v if best is None else torch.cat([best, v], 1)
        out.append(torch.topk(best, k, dim=1, largest=False, sorted=True).values.clamp_(min=0.0))
    return dict(ids=None, d2=torch.cat(out))
