"""The plain FP32 search of integer rows takes its keys from an exact 8-bit copy: ids, distances and counts
equal the oracle's for queries the copy holds and for those it does not (fractions, also ones that vanish
when the copy's offset is subtracted, values outside its range), with 1, 2 and 4 warps per query, pools in
both memories, and on loaded graphs."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d, lo", [(1, 0), (32, -100), (100, 0), (128, 7), (258, -255)])
def test_int_rows_equal_oracle(nsg, d, lo):
    rng = np.random.default_rng(d)
    n, R, k, L = 2000, 24, 10, 50
    base = (rng.integers(0, 256, (n, d)) + lo).astype(np.float32)
    base[0], base[1] = lo, lo + 255
    adj = rng.integers(0, n, (n, R)).astype(np.int32)
    q = (rng.integers(0, 256, (60, d)) + lo).astype(np.float32)
    q[0::4, 0] += 0.5
    q[1::4, d // 2] = lo + 300
    q[2::8, d - 1] = 1e-9
    idx = nsg.nsg_index_from_graph(torch.from_numpy(base).cuda(), torch.from_numpy(adj).cuda(), 5)
    rid, rd2, rexp, _ = oracle.search(adj, base, 5, q, k, L)
    for w in (1, 2, 4):
        for pool in (1, 2):
            out = idx.search_ex(torch.from_numpy(q).cuda(), k, L,
                                params=nsg.SearchParams(warps_per_query=w, pool=pool))
            ids, d2 = out["ids"].cpu().numpy(), out["d2"].cpu().numpy()
            whole = (q == np.rint(q)).all(1)  # the fractions' distances round
            assert np.array_equal(out["n_expand"].cpu().numpy()[whole], rexp[whole])
            assert np.array_equal(ids[whole], rid[whole])
            assert np.array_equal(d2[whole], rd2[whole])
            assert np.allclose(d2[~whole], rd2[~whole], rtol=1e-5)
