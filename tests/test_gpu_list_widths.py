"""Re-ranked lists of every width class above 128 entries, and both edges of the widest ones:
screened lists of 129 to 256 entries in the exact form (k + 16) and by re-rank width.  Small
integer values, so keys and distances are exact in every form and the lists equal the
oracle's bit for bit (ties by id)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_10135_gb300 import ann, build
from tests.parity import as_u32

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    ann.lib()
    ann.device_status()
    yield
    assert ann.device_status() == 0


def _ints(n, d, seed):
    return np.random.default_rng(seed).integers(-2, 3, size=(n, d)).astype(np.float32)


@pytest.mark.parametrize("kind", ["f32", "f16"])
@pytest.mark.parametrize("precision,k,rerank_k",
                         [(ann.EXACT, k, 0) for k in (113, 145, 177, 208, 209, 224, 239, 240)] +
                         [(ann.EXACT, 64, 225), (ann.F16_RERANK, 64, 240),
                          (ann.BF16_RERANK, 200, 255)])
def test_shard_lists(kind, precision, k, rerank_k):
    n, d = 900, 24
    X = _ints(n, d, k + rerank_k)
    Xt = torch.from_numpy(X).to(DEV)
    if kind == "f16":
        Xt = Xt.half()
    mem = np.concatenate([np.arange(n), np.arange(0, n, 3), [5]]).astype(np.uint32)
    off = np.array([0, n, n + 300, n + 301], dtype=np.int64)
    ids, dist = ann.shard_knn(Xt, torch.from_numpy(mem.view(np.int32)).to(DEV),
                              torch.from_numpy(off).to(DEV), k, precision, rerank_k)
    oi, od = oracle.shard_knn(X, mem, off, k)
    assert np.array_equal(as_u32(ids), oi)
    assert np.array_equal(dist.cpu().numpy().astype(np.float64), od)


@pytest.mark.parametrize("k", [209, 224, 239])
def test_queries(k):
    X, Q = _ints(1200, 24, k), _ints(70, 24, k + 1)
    ids, dist = ann.knn_query(torch.from_numpy(X).to(DEV), torch.from_numpy(Q).to(DEV), k)
    oi, od = oracle.bruteforce(X, Q, k)
    assert np.array_equal(as_u32(ids), oi)
    assert np.array_equal(dist.cpu().numpy().astype(np.float64), od)


@pytest.mark.parametrize("rerank_k", [225, 255])
def test_screened_lists(rerank_k):
    n = 600
    X = _ints(n, 24, rerank_k)
    mem = torch.arange(n, dtype=torch.int32, device=DEV)
    off = torch.tensor([0, n], dtype=torch.int64, device=DEV)
    ids, dist = ann.shard_knn_screen(torch.from_numpy(X).to(DEV), mem, off, 64, ann.EXACT,
                                     rerank_k)
    oi, od = oracle.shard_knn(X, np.arange(n, dtype=np.uint32), np.array([0, n], np.int64),
                              rerank_k)
    assert np.array_equal(as_u32(ids), oi)
    assert np.array_equal(dist.cpu().numpy().astype(np.float64), od)
