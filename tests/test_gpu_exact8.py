"""Builds on integer rows, whose distances go through an exact 8-bit copy, at the edges of the rule that
makes one: the widest rows it takes and the first it does not, spans of 255 and 256, negative offsets,
rows of one value and of no multiple of 16.  The graph equals the oracle's."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d, lo, span", [(258, -100, 255), (259, 0, 200), (17, 5, 255), (32, 0, 256), (48, -300, 255),
                                         (1, 0, 255), (130, 0, 3)])
def test_build_equals_oracle(nsg, d, lo, span):
    rng = np.random.default_rng(100 * d + span)
    centre = rng.integers(0, span + 1, (12, d))
    base = np.clip(centre[rng.integers(0, 12, 1500)] + rng.integers(-40, 41, (1500, d)), 0, span)
    base[0], base[1] = 0, span
    base = (base + lo).astype(np.float32)
    K, L, R, C = 24, 30, 20, 120
    ref = oracle.build(base, K, L, R, C, seed=0)
    idx = nsg.nsg_build(torch.from_numpy(base).cuda(), K, L, R, C, seed=0)
    adj, deg = idx.graph()
    assert idx.info()["nav"] == ref["nav"]
    assert np.array_equal(adj.cpu().numpy(), ref["adj"])
    assert np.array_equal(deg.cpu().numpy(), ref["deg"])
