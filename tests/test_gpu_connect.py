"""The connectivity pass (Alg. 2, Section 3.5 iv) on graphs where its batches
have to resolve dependent fix-ups, against the oracle's sequential loop: large
unreached components (labels over many levels), chains of fix-ups that attach
to one another, sources that fill up inside a batch, the degree fallback."""
import numpy as np
import pytest
import torch

import oracle
from paper_1707_00143_gb300 import datagen

pytestmark = pytest.mark.gpu


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def H(t):
    return t.cpu().numpy()


def graph(kind, n, R, rng):
    """Adjacency [n][R] and degrees with room left for some fix-ups."""
    adj = np.full((n, R), -1, np.int32)
    deg = np.zeros(n, np.int32)
    if kind == "paths":       # 16 disjoint paths: one long component after another
        for v in range(n - 1):
            if (v + 1) % (n // 16):
                adj[v, 0], deg[v] = v + 1, 1
    elif kind == "clusters":  # random edges inside groups of 40 ids
        for v in range(n):
            g0 = v // 40 * 40
            t = rng.choice(np.arange(g0, min(g0 + 40, n)), size=min(R - 1, 2), replace=False)
            t = t[t != v]
            adj[v, :len(t)], deg[v] = t, len(t)
    elif kind == "reversed":  # v -> v - 1: the smallest unreached id reaches nothing
        for v in range(1, n):
            adj[v, 0], deg[v] = v - 1, 1
    return adj, deg


@pytest.mark.parametrize("kind,n,d,R,L", [("empty", 700, 8, 3, 12), ("empty", 1500, 32, 40, 40),
                                          ("paths", 5000, 16, 2, 10), ("clusters", 6000, 24, 3, 20),
                                          ("reversed", 900, 12, 2, 8), ("clusters", 1200, 600, 40, 16)])
def test_connect_equals_sequential_loop(nsg, kind, n, d, R, L):
    rng = np.random.default_rng(n + R)
    base = datagen.uniform_int(n, d, seed=n, hi=64)
    adj, deg = graph(kind, n, R, rng)
    radj, rdeg, radded = oracle.connect(adj, deg, base, 5, L=L)
    a, g = T(adj), T(deg)
    added = nsg.nsg_connect(T(base), a, g, 5, L)
    assert added == len(radded)
    assert np.array_equal(H(g), rdeg)
    assert np.array_equal(H(a), radj)


def test_connect_out_of_room(nsg):
    base = datagen.uniform_int(60, 8, seed=3, hi=64)
    adj = np.full((60, 1), -1, np.int32)
    deg = np.zeros(60, np.int32)
    adj[:2, 0], deg[:2] = [1, 0], 1  # the reached pair is full
    with pytest.raises(nsg.NsgError) as e:
        nsg.nsg_connect(T(base), T(adj), T(deg), 0, 4)
    assert e.value.status == nsg.NSG_EDEGREE
