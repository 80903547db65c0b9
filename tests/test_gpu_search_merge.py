"""The search's list merge and 16-byte row reads at their edges: list widths around whole
warps, rows that cannot be read 16 bytes at a time, duplicate vectors (ties by id), an
out-degree above 32, against the oracle's search."""
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


@pytest.mark.parametrize("dtype,d,R,Ls", [(np.uint8, 128, 32, 64), (np.uint8, 20, 40, 33),
                                          (np.float32, 96, 16, 10), (np.float32, 33, 7, 100),
                                          (np.float32, 4, 64, 256)])
def test_search_equals_oracle(dtype, d, R, Ls):
    rng = np.random.default_rng(d + Ls)
    N, nq = 1500, 40
    X = rng.integers(0, 6, size=(N, d)).astype(dtype)
    X[N // 2:] = X[:N - N // 2]  # every vector twice
    Q = rng.integers(0, 6, size=(nq, d)).astype(dtype)
    deg = rng.integers(1, R + 1, size=N).astype(np.uint32)
    graph = np.full((N, R), 0xFFFFFFFF, dtype=np.uint32)
    for u in range(N):
        graph[u, :deg[u]] = rng.choice(N, size=deg[u], replace=False)
    t = lambda a: torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).to(DEV)
    ids, cnt = ann.search(t(graph), t(deg), t(X), t(Q), 3, Ls)
    oi, oc = oracle.search(graph, deg, X, Q, 3, Ls)
    assert np.array_equal(as_u32(ids), oi)
    assert np.array_equal(as_u32(cnt), oc)
