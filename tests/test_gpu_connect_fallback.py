"""The connectivity pass where most fix-ups find no room in their pools and take the smallest reached id with
a slot: many in one batch, sources that fill up among them, ids that become eligible inside the batch, and
room that pool proposals take away.  Equal to the oracle's sequential loop, and no batch for each of them."""
import numpy as np
import pytest
import torch

import oracle
from paper_1707_00143_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, R, L, free, unreached, seed", [
    (1500, 4, 6, 0.02, 0.4, 1), (1500, 4, 6, 0.3, 0.4, 2), (3000, 2, 4, 0.05, 0.3, 3), (3000, 8, 3, 0.5, 0.5, 4),
    (6000, 3, 10, 0.01, 0.2, 5), (2500, 5, 1, 0.1, 0.6, 6), (5000, 4, 20, 0.001, 0.1, 7)])
def test_equals_sequential_loop(nsg, n, R, L, free, unreached, seed):
    rng = np.random.default_rng(seed)
    base = datagen.uniform_int(n, 8, seed=seed, hi=64)
    lone = rng.random(n) < unreached  # nothing links to these; they link anywhere, some among themselves
    lone[5] = False
    others, lones = np.flatnonzero(~lone), np.flatnonzero(lone)
    adj = np.full((n, R), -1, np.int32)
    deg = np.full(n, R, np.int32)
    deg[rng.random(n) < free] -= 1
    deg[lones[rng.random(len(lones)) < 0.9]] -= 1
    ring = rng.permutation(others)
    for i, v in enumerate(ring):  # a cycle through the others keeps them reached
        adj[v, 0] = ring[(i + 1) % len(ring)]
        if deg[v] > 1:
            adj[v, 1:deg[v]] = rng.choice(others, deg[v] - 1, replace=False)
    for v in lones:
        pick = np.where(rng.random(deg[v]) < 0.2, rng.choice(lones, deg[v]), rng.choice(others, deg[v]))
        adj[v, :deg[v]] = pick
    radj, rdeg, radded = oracle.connect(adj, deg, base, 5, L=L)
    a, g = torch.from_numpy(adj).cuda(), torch.from_numpy(deg).cuda()
    added = nsg.nsg_connect(torch.from_numpy(base).cuda(), a, g, 5, L)
    assert added == len(radded)
    assert np.array_equal(g.cpu().numpy(), rdeg)
    assert np.array_equal(a.cpu().numpy(), radj)


def test_fallbacks_share_batches(nsg):
    torch.manual_seed(20000)
    base = torch.rand((20000, 16), device="cuda")
    ms = min(nsg.nsg_build(base, 5, 20, 5, 20).info()["ms_connect"] for _ in range(3))
    assert ms < 40  # 961 fix-ups, most by fallback: 132 ms with a batch for each, 22 one after the other
