"""Calls on a GPU whose memory is nearly taken: what a call can do without (the exact kNN's pre-pass, rings
and splits; a build's logs and 8-bit copy) is left out instead of failing it, with the same results."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


class Taken:
    """All of the GPU's memory but `left` bytes, while entered."""

    def __init__(self, left):
        self.left = left

    def __enter__(self):
        torch.cuda.synchronize()
        free, _ = torch.cuda.mem_get_info()
        self.held = torch.empty(free - self.left, dtype=torch.uint8, device="cuda")

    def __exit__(self, *_):
        del self.held
        torch.cuda.empty_cache()


def test_knn_query_without_scratch(nsg):
    torch.manual_seed(1)
    base = torch.randint(0, 256, (130_000, 16), device="cuda").float()
    q = torch.randint(0, 256, (200_000, 16), device="cuda").float()
    want = nsg.nsg_knn_query(base, q, 100)
    torch.cuda.empty_cache()
    spare = [torch.empty_like(t) for t in want]  # cached for the outputs
    del spare
    with Taken(160 << 20):
        got = nsg.nsg_knn_query(base, q, 100)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_build_without_logs_and_copy(nsg):
    torch.manual_seed(2)
    base = torch.randint(0, 256, (66_000, 16), device="cuda").float()
    args = (30, 40, 16, 4096)  # candidate lists of 2 GiB
    want = nsg.nsg_build(base, *args)
    adj, deg = want.graph()
    info = want.info()
    want.free()
    # the lists, ~30 MB of base, graphs and counters, and less than the 256 MB that the copy leaves free
    with Taken((2 << 30) + (200 << 20)):
        idx = nsg.nsg_build(base, *args)
        assert idx.info()["nav"] == info["nav"]
        assert idx.info()["device_bytes"] == info["device_bytes"] - 66_000 * 16  # without the 8-bit copy
    a, d = idx.graph()
    assert torch.equal(a, adj) and torch.equal(d, deg)
