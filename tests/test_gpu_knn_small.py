"""Exact kNN on short bases, on both sides of the lines that choose its kernel: base sizes, query counts
and list sizes around them, ragged; integer rows, so ids and distances equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, nq, d, k", [(8447, 33, 32, 10), (8448, 33, 32, 10), (8500, 32, 20, 1), (129, 300, 128, 100),
                                         (9000, 1025, 48, 100), (9000, 1024, 48, 100), (11000, 4097, 16, 10),
                                         (16385, 4097, 16, 3)])
def test_query_equals_oracle(nsg, n, nq, d, k):
    rng = np.random.default_rng(n + nq)
    base = rng.integers(0, 256, (n, d)).astype(np.float32)
    q = rng.integers(0, 256, (nq, d)).astype(np.float32)
    ids, d2 = nsg.nsg_knn_query(torch.from_numpy(base).cuda(), torch.from_numpy(q).cuda(), k)
    rows = rng.choice(nq, min(nq, 60), replace=False)
    rid, rd2 = oracle.knn_query(base, q[rows], k)
    assert np.array_equal(ids.cpu().numpy()[rows], rid)
    assert np.array_equal(d2.cpu().numpy()[rows], rd2)
