"""Search-and-collect through logs, whose length follows the searches seen so far: a first slice whose logs
fill, slices of a few nodes, searches longer than any log (merged lists take over), against the lists that
are merged as the searches go, bit for bit.  And logs are not slower than those lists where searches
measure most of what they meet (uniform rows: ~0.6 L K keys each; logs of half L K filled twice and took 2.2 times
as long).  The call for some nodes only keeps to the lists: it would pay for the logs each time."""
import time

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def collect(nsg, monkeypatch, engine, log, *args, **kw):
    monkeypatch.setenv("NSG_COLLECT_ENGINE", engine)
    if log:
        monkeypatch.setenv("NSG_COLLECT_LOG", log)
    return [t.cpu().numpy() for t in nsg.nsg_collect(*args, **kw)]


@pytest.mark.parametrize("d, span, K, L, C, log", [
    (32, 256, 32, 32, 100, "200000,1024"),   # logs of 1,024 keys fill, slices of 195 nodes
    (32, 256, 31, 33, 500, "5000000,1056"),  # one slice of logs that fill, the rest in one
    (32, 256, 32, 32, 100, "1100,32"),       # a node at a time, then logs longer than the space
    (128, 2, 100, 40, 500, "3000000,4000"),  # thousands of ties
    (20, 256, 200, 30, 511, ""),             # the library's own lengths
    (32, 256, 256, 128, 300, ""),            # searches longer than any log
    (600, 16, 64, 60, 300, "500000,0"),
    (4, 256, 3, 1, 5, "10000,0"),
])
def test_logs_equal_merged_lists(nsg, monkeypatch, d, span, K, L, C, log):
    rng = np.random.default_rng(7 * K + L)
    n = 6000
    base = torch.from_numpy(rng.integers(0, span, (n, d)).astype(np.float32)).cuda()
    knn = torch.from_numpy(rng.integers(0, n, (n, K)).astype(np.int32)).cuda()
    want = collect(nsg, monkeypatch, "merge", "", base, knn, 17, L, C, v0=11, nv=3001)
    got = collect(nsg, monkeypatch, "log", log, base, knn, 17, L, C, v0=11, nv=3001)
    for w, g in zip(want, got):
        assert np.array_equal(w, g)


def test_build_log_no_slower_than_merged_lists(nsg, monkeypatch):
    torch.manual_seed(1)
    base = torch.rand((20000, 16), device="cuda")

    def ms(engine):
        monkeypatch.setenv("NSG_COLLECT_ENGINE", engine)
        return min(nsg.nsg_build(base, 100, 60, 50, 500).info()["ms_collect"] for _ in range(4))

    assert ms("log") < 1.15 * ms("merge")


def test_collect_call_pays_for_no_logs(nsg, monkeypatch):
    rng = np.random.default_rng(5)
    base = torch.from_numpy(rng.standard_normal((20000, 96)).astype(np.float32)).cuda()
    blocks = rng.integers(0, 25, (20000, 20)) + np.arange(20000)[:, None] // 25 * 25  # short searches
    knn = torch.from_numpy(blocks.astype(np.int32)).cuda()

    def seconds(engine):
        if engine:
            monkeypatch.setenv("NSG_COLLECT_ENGINE", engine)
        best = 1e9
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            nsg.nsg_collect(base, knn, 17, 500, 500, v0=0, nv=5000)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    default = seconds("")
    assert default < 1.3 * seconds("merge")
