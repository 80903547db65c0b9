"""Candidate pools of the tile sweep where they can go wrong: more ties at the k'-th key
than a compaction may keep, every list width class up to the widest, keys on both sides
of zero, shards of one row and of odd sizes.  Integer values, so every form's keys and
distances are exact and the lists equal the oracle's bit for bit (ties by id)."""
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


def _data(kind, n, d, rng):
    if kind == "equal":
        return np.full((n, d), 3, dtype=np.uint8)
    if kind == "levels":  # few distinct vectors: thousands of ties at any rank
        return rng.integers(0, 2, size=(n, 1), dtype=np.uint8).repeat(d, 1)
    return rng.integers(0, 4, size=(n, d), dtype=np.uint8)


def _shards(n, sizes, rng):
    mem = [np.sort(rng.choice(n, size=s, replace=False)).astype(np.uint32) for s in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return np.concatenate(mem), off


@pytest.mark.parametrize("kind", ["equal", "levels", "small"])
@pytest.mark.parametrize("k", [1, 31, 64, 129, 240])
def test_ties_and_list_widths(kind, k):
    rng = np.random.default_rng(k)
    n, d = 3001, 16
    X = _data(kind, n, d, rng)
    mem, off = _shards(n, [1, 3001, 257, 130], rng)
    ids, dist = ann.shard_knn(torch.from_numpy(X).to(DEV), torch.from_numpy(mem.view(np.int32)).to(DEV),
                              torch.from_numpy(off).to(DEV), k)
    oi, od = oracle.shard_knn(X, mem, off, k)
    assert np.array_equal(as_u32(ids), oi)
    assert np.array_equal(dist.cpu().numpy().astype(np.float64), od)


@pytest.mark.parametrize("precision,k,rerank_k", [(ann.EXACT, 60, 0), (ann.EXACT, 64, 200),
                                                  (ann.F16_RERANK, 64, 256),
                                                  (ann.F16_RERANK, 33, 128),
                                                  (ann.BF16_RERANK, 64, 160)])
def test_screened_lists_with_keys_across_zero(precision, k, rerank_k):
    # values -2 .. 2: |y|^2 / 2 - x.y takes both signs, most of them many times over
    rng = np.random.default_rng(rerank_k + k)
    n, d = 2500, 24
    X = rng.integers(-2, 3, size=(n, d)).astype(np.float32)
    mem, off = _shards(n, [2500, 1, 300], rng)
    ids, dist = ann.shard_knn(torch.from_numpy(X).to(DEV), torch.from_numpy(mem.view(np.int32)).to(DEV),
                              torch.from_numpy(off).to(DEV), k, precision, rerank_k)
    oi, od = oracle.shard_knn(X, mem, off, k)
    assert np.array_equal(as_u32(ids), oi)
    assert np.array_equal(dist.cpu().numpy().astype(np.float64), od)
