"""Which rows get the 8-bit copy that plain searches of integer rows use (the index's bytes tell), and that
making it does not take longer than reading the rows: padded rows whose zeros are no values, the span's ends,
one fraction or NaN anywhere, values past 2^24."""
import time

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d, lo, span, odd, copy", [
    (1, 5, 255, None, True), (3, 40, 255, None, True), (17, -300, 255, None, True), (130, 7, 255, None, True),
    (32, 2**24, 254, None, True),
    (32, 2**24, 255, None, False),  # 2^24 + 255 rounds to a span of 256
    (258, -100, 255, None, True), (259, 0, 200, None, False), (32, 0, 256, None, False),
    (33, 10, 200, 0.5, False), (33, 10, 200, np.nan, False), (20, 10, 200, np.inf, False), (20, 3, 0, None, True)])
def test_copy_made_and_right(nsg, d, lo, span, odd, copy):
    rng = np.random.default_rng(d)
    n, R = 2500, 12
    base = (rng.integers(0, span + 1, (n, d)) + lo).astype(np.float32)
    base[0], base[1] = lo, lo + span
    if lo == 2**24:  # FP32 holds every second integer here
        base = (base // 2 * 2).astype(np.float32)
    if odd is not None:
        base[n - 1, d - 1] = odd
    adj = rng.integers(0, n, (n, R)).astype(np.int32)
    idx = nsg.nsg_index_from_graph(torch.from_numpy(base).cuda(), torch.from_numpy(adj).cuda(), 5)
    plain = 4 * n * ((d + 3) // 4 * 4 + R + 1) + 16  # rows, graph, degrees, flags
    assert idx.info()["device_bytes"] - plain == (n * ((d + 15) // 16 * 16) if copy else 0)
    if odd is None or np.isfinite(odd):
        q = base[rng.choice(n, 40, replace=False)].copy()
        ids, d2 = idx.search(torch.from_numpy(q).cuda(), 10, 60)
        rid, rd2, _, _ = oracle.search(adj, base, 5, q, 10, 60)
        if odd is None:
            assert np.array_equal(ids.cpu().numpy(), rid) and np.array_equal(d2.cpu().numpy(), rd2)


def test_copy_costs_a_read(nsg):
    n, d = 1_000_000, 128
    base = torch.randint(0, 256, (n, d), device="cuda").float()
    adj = torch.zeros((n, 1), dtype=torch.int32, device="cuda")
    deg = torch.ones(n, dtype=torch.int32, device="cuda")

    def seconds(b):
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            idx = nsg.nsg_index_from_graph(b, adj, 0, deg)
            best = min(best, time.perf_counter() - t0)
            idx.free()
        return best

    whole = seconds(base)
    base[0, 0] = 0.5
    assert whole - seconds(base) < 0.6e-3  # 1.0 ms a value at a time


def test_prepared_copy_is_the_same_one(nsg):
    rng = np.random.default_rng(1)
    base = torch.from_numpy(rng.integers(-50, 200, (4000, 40)).astype(np.float32)).cuda()
    adj = torch.from_numpy(rng.integers(0, 4000, (4000, 16)).astype(np.int32)).cuda()
    idx = nsg.nsg_index_from_graph(base, adj, 3)
    q = base[:300].contiguous()
    want = idx.search(q, 10, 50)
    before = idx.info()["device_bytes"]
    idx.prepare(nsg.PREC_U8)
    info = idx.info()
    assert info["device_bytes"] == before
    out = idx.search_ex(q, 10, 50, params=nsg.SearchParams(precision=nsg.PREC_U8))
    assert torch.equal(out["ids"], want[0]) and torch.equal(out["d2"], want[1])
    idx.free()
