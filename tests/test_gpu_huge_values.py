"""Selections among keys whose range passes FP32's: two clusters on opposite sides of zero,
squared distances within one finite, tile keys across both up to +inf.  The search among a
pool's keys has to end, and the lists are those of the oracle by the float rule."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_10135_gb300 import ann, build
from tests.parity import check_float_lists

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    ann.lib()
    ann.device_status()
    yield
    ann.tile_prune(True)
    assert ann.device_status() == 0


# |x|^2 = 1.6e38: keys from -0.8e38 to 2.5e38, all finite, their difference not;
# |x|^2 = 2.4e38: keys to the other cluster are +inf
def _data(a, spread, n, seed):
    rng = np.random.default_rng(seed)
    u = np.ones(8) / np.sqrt(8.0)
    side = np.where(np.arange(n) % 2 == 0, 1.0, -1.0)[:, None]
    X = (a * (side * u + spread * rng.normal(size=(n, 8)).clip(-2, 2))).astype(np.float32)
    assert np.isfinite((X * X).sum(axis=1, dtype=np.float32)).all()
    return X


@pytest.mark.parametrize("a,spread", [(1.25e19, 0.06), (1.55e19, 0.04)])
@pytest.mark.parametrize("k", [40, 100])
def test_queries(a, spread, k):
    X, Q = _data(a, spread, 1500, k), _data(a, spread, 100, k + 1)
    ids, dist = ann.knn_query(torch.from_numpy(X).to(DEV), torch.from_numpy(Q).to(DEV), k)
    torch.cuda.synchronize()
    oi, od = oracle.bruteforce(X, Q, k)
    check_float_lists(np.concatenate([X, Q]), range(1500, 1600), ids, dist.cpu().numpy(), oi, od)


@pytest.mark.parametrize("a,spread", [(1.25e19, 0.06), (1.55e19, 0.04)])
def test_shard_lists(a, spread):
    n, k = 1500, 40
    X = _data(a, spread, n, 7)
    mem, off = np.arange(n, dtype=np.uint32), np.array([0, n], dtype=np.int64)
    ann.tile_prune(False)
    ids, dist = ann.shard_knn(torch.from_numpy(X).to(DEV), torch.from_numpy(mem.view(np.int32)).to(DEV),
                              torch.from_numpy(off).to(DEV), k)
    torch.cuda.synchronize()
    oi, od = oracle.shard_knn(X, mem, off, k)
    check_float_lists(X, range(n), ids, dist.cpu().numpy(), oi, od)
