"""Navigating node vs the CPU oracle where the kernel's blocks end: rows of one value, of a tile of 64 and
one more, wider; adjacency rows of more than the 128 neighbours taken at a time; pools of 1 and 1,024;
rows that repeat ids or end early.  FP64 in a stated order: the same node.  NaN distances have no order:
the start node stays first."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d, K, L", [(1, 5, 10), (63, 20, 40), (64, 128, 40), (65, 129, 1), (100, 300, 200),
                                     (700, 100, 33), (12, 64, 1024)])
def test_navigate_equals_oracle(nsg, d, K, L):
    rng = np.random.default_rng(10 * d + K)
    n = 3000
    base = rng.standard_normal((n, d)).astype(np.float32)
    knn = rng.integers(0, n, (n, K)).astype(np.int32)
    knn[::5, K // 2:] = -1
    c = oracle.centroid(base)
    for start in (0, 1234, n - 1):
        nav = nsg.nsg_navigate(torch.from_numpy(base).cuda(), torch.from_numpy(knn).cuda(),
                               torch.from_numpy(c).cuda(), start, L)
        assert nav == oracle.navigate(knn, base, c, start, L)


def test_navigate_nan(nsg):
    rng = np.random.default_rng(3)
    base = rng.standard_normal((500, 20)).astype(np.float32)
    base[:, 7] = np.nan
    knn = torch.from_numpy(rng.integers(0, 500, (500, 30)).astype(np.int32)).cuda()
    assert nsg.nsg_navigate(torch.from_numpy(base).cuda(), knn, torch.zeros(20, dtype=torch.float64).cuda(), 321,
                            16) == 321
