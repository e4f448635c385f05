"""Tensor-core kNN where its pre-pass bounds the rows, the base is split over
the SMs and the rings fill: integer data, so ids and distances equal the
oracle's bit for bit.  Ties (few distinct values) meet the bound itself;
ragged rows leave row groups empty; k = 256 fills the longest lists."""
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


@pytest.mark.parametrize("n,d,k,hi", [(6001, 32, 10, 256), (5000, 16, 20, 3), (9000, 100, 64, 256),
                                      (40007, 24, 5, 16)])
def test_self_join_with_bound(nsg, n, d, k, hi):
    base = datagen.uniform_int(n, d, seed=n, hi=hi)
    ids, d2 = nsg.nsg_knn_init(T(base), k)
    rows = np.arange(0, n, max(1, n // 1500))
    rid, rd2 = oracle.knn_query(base, base[rows], k + 1)
    for j, r in enumerate(rows):  # the row itself is skipped by id
        assert np.array_equal(H(ids[r]), rid[j][rid[j] != r][:k])
        assert np.array_equal(H(d2[r]), rd2[j][rid[j] != r][:k])


@pytest.mark.parametrize("n,nq,d,k,hi", [(30001, 700, 100, 100, 256), (30001, 129, 64, 1, 256), (12000, 300, 128, 256, 256),
                                         (20000, 1, 33, 10, 256), (16000, 513, 20, 40, 2)])
def test_queries_split_over_the_base(nsg, n, nq, d, k, hi):
    base = datagen.uniform_int(n, d, seed=n + d, hi=hi)
    q = datagen.uniform_int(nq, d, seed=n + d + 1, hi=hi)
    ids, d2 = nsg.nsg_knn_query(T(base), T(q), k)
    rid, rd2 = oracle.knn_query(base, q, k)
    assert np.array_equal(H(d2), rd2)
    assert np.array_equal(H(ids), rid)
