"""Search-and-collect vs the CPU oracle where its two forms meet their edges: logs that overflow and
are compacted (random adjacency: nearly every neighbour is new), every block size of the selection,
lists longer than what is measured, equal distances by the thousand, rows wider than 512 values, and
the pool and degree from which the lists are merged instead.  Integer data: equal bit for bit."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

N = 6000


@pytest.mark.parametrize("d, span, K, L, C", [
    (32, 256, 32, 32, 100),    # log of 1,024 keys, overflows
    (32, 256, 31, 33, 500),    # log of 1,056, overflows with more to keep
    (128, 2, 100, 40, 500),    # few distances: thousands of ties at the bound
    (32, 1, 40, 24, 100),      # one distance
    (4, 256, 3, 1, 5),         # the smallest searches
    (20, 256, 200, 30, 511),   # 256 threads per node
    (32, 256, 30, 60, 4096),   # 512 threads; fewer keys than the list holds
    (600, 16, 64, 60, 300),    # wide rows
    (32, 256, 128, 128, 300),  # log of 8,192
    (32, 256, 256, 128, 300),  # the longest log
    (32, 256, 257, 128, 300),  # merged lists
])
def test_collect_equals_oracle(nsg, d, span, K, L, C):
    rng = np.random.default_rng(1000 * K + L)
    base = rng.integers(0, span, (N, d)).astype(np.float32)
    knn = rng.integers(0, N, (N, K)).astype(np.int32)
    if K > 40:
        knn[::7, K // 2:] = -1
    nav, v0, nv = 17, 11, 3001
    ids, d2, cnt, st = nsg.nsg_collect(torch.from_numpy(base).cuda(), torch.from_numpy(knn).cuda(), nav, L, C, v0=v0,
                                       nv=nv)
    ids, d2, cnt = ids.cpu().numpy(), d2.cpu().numpy(), cnt.cpu().numpy()
    assert (st.cpu().numpy() == 0).all()
    for j in [0, 1, nav - v0, nv - 1, *rng.choice(nv, 30, replace=False)]:
        rid, rd2, rc, _, _ = oracle.collect(knn, base, nav, int(v0 + j), L, C)
        assert cnt[j] == rc, j
        assert np.array_equal(ids[j], rid), j
        assert np.array_equal(d2[j], rd2), j
