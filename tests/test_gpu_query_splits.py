"""Ground-truth queries whose columns are split over CTAs: one query, ragged last ranges,
ranges shorter than the list, ties across ranges, every width of the vectorised uint8
gather and the general one beside it."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_10135_gb300 import ann, build
from tests.parity import as_u32, check_float_lists

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    ann.lib()
    ann.device_status()
    yield
    assert ann.device_status() == 0


def _run(X, Q, k):
    ids, dist = ann.knn_query(torch.from_numpy(X).to(DEV), torch.from_numpy(Q).to(DEV), k)
    return as_u32(ids), dist.cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("N,nq,d,k", [(1, 1, 16, 1), (257, 3, 64, 10), (5000, 1, 128, 100),
                                      (40_001, 129, 48, 10), (9_999, 1000, 208, 1),
                                      (3_000, 5, 240, 240), (2_600, 300, 130, 64)])
def test_u8_queries(N, nq, d, k):
    rng = np.random.default_rng(N + d)
    X = rng.integers(0, 256 if d > 100 else 3, size=(N, d), dtype=np.uint8)
    Q = rng.integers(0, 256 if d > 100 else 3, size=(nq, d), dtype=np.uint8)
    ids, dist = _run(X, Q, k)
    oi, od = oracle.bruteforce(X, Q, k)
    assert np.array_equal(ids, oi)
    assert np.array_equal(dist, od)


@pytest.mark.parametrize("N,nq,d,k", [(20_003, 2, 75, 10), (7_000, 260, 96, 100), (300, 1, 33, 1)])
def test_f32_queries(N, nq, d, k):
    rng = np.random.default_rng(N)
    X = rng.normal(size=(N, d)).astype(np.float32)
    Q = rng.normal(size=(nq, d)).astype(np.float32)
    ids, dist = _run(X, Q, k)
    oi, od = oracle.bruteforce(X, Q, k)
    XQ = np.concatenate([X, Q])  # the rule takes the row's own vector from one array
    check_float_lists(XQ, range(N, N + nq), ids, dist, oi, od)
