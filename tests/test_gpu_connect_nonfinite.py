"""The connectivity pass on rows with NaN and infinite values, whose distances sort after the finite ones
(infinity, then NaN, ties by id): the graph of the sequential loop, restated here."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def rank(base, u):
    with np.errstate(all="ignore"):
        d = ((base - base[u]) ** 2).sum(1)
    kind = np.where(np.isnan(d), 2, np.where(np.isinf(d), 1, 0))
    return [(int(k), float(x) if k == 0 else 0.0, i) for i, (k, x) in enumerate(zip(kind, d))]


def search(adj, key, nav, L):
    pool, seen, done = [key[nav]], {nav}, set()
    while True:
        nxt = next((e[2] for e in pool if e[2] not in done), -1)
        if nxt < 0:
            return [e[2] for e in pool]
        done.add(nxt)
        for v in adj[nxt]:
            if v not in seen:
                seen.add(v)
                pool.append(key[v])
        pool = sorted(pool)[:L]


def connect(adj, base, nav, L, R):
    n, reached = len(adj), set()

    def reach(v):
        stack = [v]
        while stack:
            x = stack.pop()
            if x not in reached:
                reached.add(x)
                stack += adj[x]

    reach(nav)
    for u in range(n):
        if u in reached:
            continue
        pool = search(adj, rank(base, u), nav, L)
        s = next((v for v in pool if len(adj[v]) < R), None)
        if s is None:
            s = min(v for v in reached if len(adj[v]) < R)
        adj[s].append(u)
        reach(u)


@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("bad", ["nan", "inf", "both"])
def test_equals_sequential_loop(nsg, bad, seed):
    rng = np.random.default_rng(seed)
    n, R, L, d = 400, 5, 6, 4
    base = rng.integers(0, 8, (n, d)).astype(np.float32)
    rows = rng.permutation(n)
    if bad != "inf":
        base[rows[:60], 1] = np.nan
    if bad != "nan":
        base[rows[60:120], 2] = np.inf
    adj = np.full((n, R), -1, np.int32)
    deg = rng.integers(0, 3, n).astype(np.int32)  # sparse: most nodes are unreached
    for v in range(n):
        adj[v, :deg[v]] = rng.choice(n, deg[v], replace=False)
    want = [adj[v, :deg[v]].tolist() for v in range(n)]
    connect(want, base, 7, L, R)
    a, g = torch.from_numpy(adj).cuda(), torch.from_numpy(deg).cuda()
    nsg.nsg_connect(torch.from_numpy(base).cuda(), a, g, 7, L)
    a, g = a.cpu().numpy(), g.cpu().numpy()
    assert [a[v, :g[v]].tolist() for v in range(n)] == want
