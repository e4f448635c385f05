"""Both tensor-core kNN kernels over the forms a call can take, whichever the sizes would choose: float rows
and their re-rank, rows wider than 128 values (streamed), lists carried over chunks of the base, splits of
the base, ids only, self joins with and without the pre-pass.  Tolerances as for the chosen kernel: integer
rows equal the oracle's bit for bit, float rows' distances within 1e-5 and no neighbour farther than the
true k-th."""
import numpy as np
import pytest
import torch

import oracle
from paper_1707_00143_gb300 import datagen

pytestmark = pytest.mark.gpu


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture(params=["units", "small"])
def engine(request, monkeypatch):
    monkeypatch.setenv("NSG_KNN_ENGINE", request.param)
    return request.param


def check(ids, d2, base, q, k, rid, rd2, whole):
    ids, d2 = ids.cpu().numpy(), d2.cpu().numpy()
    if whole:
        assert np.array_equal(ids, rid) and np.array_equal(d2, rd2)
        return
    assert np.allclose(d2, rd2, rtol=1e-5, atol=0)
    exact = ((base[ids].astype(np.float64) - q[:, None, :]) ** 2).sum(-1)
    assert np.allclose(d2, exact, rtol=1e-5, atol=0)
    assert (exact <= rd2[:, -1:].astype(np.float64) * (1 + 1e-5)).all()
    assert oracle.recall(ids, rid, k) >= 0.995


@pytest.mark.parametrize("chunk", [0, 3])
@pytest.mark.parametrize("n,nq,d,k,whole", [
    (9000, 300, 96, 10, False), (9000, 33, 200, 20, False), (4000, 130, 960, 100, False), (3000, 257, 1024, 10, False),
    (20000, 40, 300, 1, False), (9000, 70, 200, 30, True), (9000, 500, 100, 64, True), (16500, 20, 128, 100, True)])
def test_query(nsg, engine, monkeypatch, n, nq, d, k, whole, chunk):
    if chunk:
        monkeypatch.setenv("NSG_KNN_CHUNK_TILES", str(chunk))
    make = datagen.uniform_int if whole else datagen.uniform_float
    base, q = make(n, d, seed=n + d), make(nq, d, seed=n + d + 1)
    ids, d2 = nsg.nsg_knn_query(T(base), T(q), k)
    rid, rd2 = oracle.knn_query(base, q, k)
    check(ids, d2, base, q, k, rid, rd2, whole)


@pytest.mark.parametrize("chunk", [0, 7])
@pytest.mark.parametrize("n,d,k,whole", [(9001, 48, 20, False), (3000, 200, 100, False), (9001, 100, 10, True),
                                         (2500, 128, 256, True), (1111, 960, 30, True), (40007, 24, 5, True)])
def test_self_join(nsg, engine, monkeypatch, n, d, k, whole, chunk):
    if chunk:
        monkeypatch.setenv("NSG_KNN_CHUNK_TILES", str(chunk))
    base = (datagen.uniform_int if whole else datagen.uniform_float)(n, d, seed=n + d)
    ids, d2 = nsg.nsg_knn_init(T(base), k)
    only, _ = nsg.nsg_knn_init(T(base), k, with_d2=False)
    assert torch.equal(only, ids)
    rows = np.arange(0, n, max(1, n // 400))
    rid, rd2 = oracle.knn_query(base, base[rows], k + 1)
    keep = rid != rows[:, None]
    keep[keep.all(1), -1] = False  # a duplicate of the row pushed it out
    rid, rd2 = rid[keep].reshape(len(rows), k), rd2[keep].reshape(len(rows), k)
    check(ids[T(rows)], d2[T(rows)], base, base[rows], k, rid, rd2, whole)


def test_both_kernels_agree_on_a_large_float_base(nsg, monkeypatch):
    base, q = datagen.uniform_float(60000, 72, seed=1), datagen.uniform_float(1000, 72, seed=2)
    out = []
    for e in ("units", "small"):
        monkeypatch.setenv("NSG_KNN_ENGINE", e)
        out.append(nsg.nsg_knn_query(T(base), T(q), 50))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


@pytest.mark.parametrize("scale", [1.0, 4096.0, 1e6, 3e19])
def test_far_queries(nsg, monkeypatch, scale):
    """Queries so far away that FP32 distances tie by the hundred (or, past FP32's range, all do): ties go by
    id in both kernels, whatever bounds the pre-pass of one of them."""
    n, d = 30000, 96
    base, q = datagen.uniform_float(n, d, seed=5), datagen.uniform_float(400, d, seed=6)
    q = (q * np.float32(scale)).astype(np.float32)
    out = []
    for e in ("units", "small"):
        monkeypatch.setenv("NSG_KNN_ENGINE", e)
        out.append([t.cpu().numpy() for t in nsg.nsg_knn_query(T(base), T(q), 10)])
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    if scale > 1e19:
        assert np.isinf(out[0][1]).all()
        assert np.array_equal(out[0][0], np.tile(np.arange(10), (400, 1)))


@pytest.mark.parametrize("d", [24, 100, 200])
def test_tied_clusters(nsg, monkeypatch, d):
    """Clusters far from the origin, whose rows round to few BF16 values: which candidates a full list keeps is
    decided by the norms' last bits, the same for both kernels."""
    rng = np.random.default_rng(d)
    n = 24000
    base = (100 * rng.standard_normal((n // 100, d))).repeat(100, 0) + rng.random((n, d))
    base = base.astype(np.float32)
    out = []
    for e in ("units", "small"):
        monkeypatch.setenv("NSG_KNN_ENGINE", e)
        out.append([t.cpu().numpy() for t in nsg.nsg_knn_query(T(base), T(base[::50] + np.float32(0.01)), 10)])
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
