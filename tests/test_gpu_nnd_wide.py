"""nn-descent's join reads offers ahead for rows of up to 256 values and one at a time for wider ones: both
sides of that line, and of the kernels' row shapes, equal the oracle's lists on integer rows."""
import numpy as np
import pytest
import torch

import oracle
from paper_1707_00143_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [256, 260, 512, 516, 1024, 1028])
def test_equals_oracle(nsg, d):
    base = datagen.uniform_int(700, d, seed=d, hi=64)
    p = nsg.NnDescentParams(20, 20, 4, 0.0, 3)  # members of up to 40 offers
    ids, d2, it, upd = nsg.nsg_knn_nndescent(torch.from_numpy(base).cuda(), 24, p)
    rid, rd2, rit, rupd = oracle.nndescent(base, 24, S=20, Sr=20, iters=4, delta=0.0, seed=3)
    assert (it, upd) == (rit, rupd)
    assert np.array_equal(ids.cpu().numpy(), rid) and np.array_equal(d2.cpu().numpy(), rd2)
