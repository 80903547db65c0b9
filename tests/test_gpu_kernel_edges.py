"""Edges of the re-rank of wide rows, of the skipping bounds' windows and of the few-centroid
assignment.  The list tests use small integers, so keys and distances are exact in every
form and the lists equal the oracle's bit for bit (ties by id); k-means sums run in sample
order in 64 bits, so centroids and shards are equal bit for bit too."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_10135_gb300 import ann, build, datagen
from tests.parity import as_u32

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    ann.lib()
    ann.device_status()
    ann.tile_prune(True)
    yield
    ann.tile_prune(True)
    assert ann.device_status() == 0


def T(a):
    return torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).to(DEV)


def _shards(n, sizes, rng):
    mem = [np.sort(rng.choice(n, size=s, replace=False)).astype(np.uint32) for s in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return np.concatenate(mem), off


# 16-byte chunks a row: 33 (one lane in its second round), 64, 65, 127, 128, and 129, which
# keeps the loop over chunks; lists of 64, 128 and 256 candidates, one shard shorter than any
@pytest.mark.parametrize("chunks", [33, 64, 65, 127, 128, 129])
@pytest.mark.parametrize("kind,kp", [("f16", 256), ("f32", 128), ("bf16", 64)])
def test_rerank_of_wide_rows(kind, kp, chunks):
    rng = np.random.default_rng(chunks + kp)
    n, d = 700, chunks * (4 if kind == "f32" else 8)
    X = rng.integers(-2, 3, size=(n, d)).astype(np.float32)
    Xt = T(X) if kind == "f32" else T(X).to(torch.float16 if kind == "f16" else torch.bfloat16)
    prec = ann.BF16_RERANK if kind == "bf16" else ann.F16_RERANK
    mem, off = _shards(n, [700, 1, 50], rng)
    ids, dist = ann.shard_knn(Xt, T(mem), T(off), 33, prec, kp)
    oi, od = oracle.shard_knn(X, mem, off, 33)
    assert np.array_equal(as_u32(ids), oi)
    assert np.array_equal(dist.cpu().numpy().astype(np.float64), od)


# shards on both sides of the window's 512 rows and of lists longer than a window's rows
@pytest.mark.parametrize("kind,prec,k,kp", [("u8", ann.EXACT, 1, 0), ("u8", ann.EXACT, 240, 0),
                                            ("f32", ann.EXACT, 32, 0),
                                            ("f32", ann.F16_RERANK, 64, 256),
                                            ("f32", ann.BF16_RERANK, 20, 100)])
def test_windows_at_shard_edges(kind, prec, k, kp):
    rng = np.random.default_rng(k + kp)
    sizes = [1, 127, 255, 257, 511, 512, 513, 1025, 6000]
    n, d = 6000, 32
    lab = rng.integers(0, 24, n)
    X = rng.integers(0, 40, size=(24, d))[lab] + rng.integers(0, 3, size=(n, d))
    X = X.astype(np.uint8 if kind == "u8" else np.float32)
    Xt = T(X)
    mem, off = _shards(n, sizes, rng)
    ann.tile_prune(False)
    a = ann.shard_knn(Xt, T(mem), T(off), k, prec, kp)
    ann.tile_prune_stats()
    ann.tile_prune(True)
    b = ann.shard_knn(Xt, T(mem), T(off), k, prec, kp)
    st = ann.tile_prune_stats()
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    assert 0 < st["swept"] <= st["tiles"]
    oi, od = oracle.shard_knn(X, mem, off, k)
    assert np.array_equal(as_u32(b[0]), oi)
    assert np.array_equal(b[1].cpu().numpy().astype(np.float64), od)


@pytest.mark.parametrize("C", [2, 3, 31, 32, 33])
@pytest.mark.parametrize("kind,d", [("u8", 20), ("f32", 100), ("f16", 72), ("bf16", 8)])
def test_few_centroids(kind, d, C):
    n, r, iters = 1037, min(3, C), 3
    if kind == "u8":
        X = datagen.clustered_u8(n, d, 9, seed=C)
        Xt = T(X)
    else:
        X = datagen.gaussian_mixture_f32(n, d, 9, 2.0, seed=C)
        X[:, 1] = 0.0
        X[:, 0] *= np.float32(1e-39 if kind == "f32" else 1e-7)  # below the smallest normal
        Xt = T(X).to(dict(f32=torch.float32, f16=torch.float16, bf16=torch.bfloat16)[kind])
        X = Xt.float().cpu().numpy() if kind != "f16" else Xt.cpu().numpy()
    sample, init_rows = datagen.kmeans_sample(n, C, C)
    init = X[init_rows].astype(np.float32)
    cent, mem, off = ann.partition(Xt, C, r, T(init), T(sample), iters)
    cent_o, _, mem_o, off_o = oracle.partition(X, init, sample, iters, C, r)
    assert np.array_equal(cent.cpu().numpy().view(np.uint32), cent_o.view(np.uint32))
    assert np.array_equal(off.cpu().numpy(), off_o)
    assert np.array_equal(as_u32(mem), mem_o)
