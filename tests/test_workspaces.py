"""Scratch that was sized for one launch and serves a smaller one: the centroid screen of a
k-means sample below the number of vectors, and queries with fewer rows than the scratch was
reported for."""
import ctypes as ct

import numpy as np
import pytest
import torch

import oracle
from paper_2605_10135_gb300 import ann, build, datagen
from tests.parity import as_u32

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def L():
    build.build()
    return ann.lib()


def _query_bytes(L, N, nq, d, dtype, k):
    n = ct.c_size_t(0)
    assert L.ann_knn_query_workspace(N, nq, d, dtype, k, ct.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("N,d,dtype,k", [(20_000, 16, 3, 10), (20_000, 32, 0, 20),
                                         (1_000_000, 128, 3, 100), (300, 16, 3, 1)])
def test_scratch_of_more_queries_serves_fewer(L, N, d, dtype, k):
    sizes = [1, 100, 129, 500, 1000, 2000, 5000, 10_000, 15_000, 40_000]
    dummy = ct.c_void_p(16)  # never dereferenced: refused by the check after the scratch check
    for i, more in enumerate(sizes):
        have = _query_bytes(L, N, more, d, dtype, k)
        for nq in sizes[:i + 1]:
            rc = L.ann_knn_query(dummy, N, dummy, nq, d, dtype, k, dummy, dummy, dummy, have, None)
            assert rc != 5, (more, nq, L.ann_last_error())
    # less than one query's scratch is refused still
    rc = L.ann_knn_query(dummy, N, dummy, 1, d, dtype, k, dummy, dummy, dummy, 4096, None)
    assert rc == 5


# (partition: vectors, with a sample of half of them; training: sample rows)
@pytest.mark.parametrize("what", ["partition", "selective", "train"])
def test_reported_scratch_grows_with_the_rows(L, what):
    sizes = [1000, 2000, 5000, 9000, 10_000, 14_000, 18_000, 20_000, 40_000, 45_000, 100_000]
    n, last = ct.c_size_t(0), 0
    p = ann._SelectiveParams(1.2, 2.0, 4096, 0, 2, 8)
    for m in sizes:  # C = 1,000: four column tiles in the centroid screen
        if what == "partition":
            rc = L.ann_partition_workspace(m, 96, 1000, 2, m // 2, ct.byref(n))
        elif what == "selective":
            rc = L.ann_partition_selective_workspace(m, 96, 1000, m // 2, ct.byref(p), ct.byref(n))
        else:
            rc = L.ann_learned_train_workspace(1_000_000, 96, 0, m, 40, 256, ct.byref(n))
        assert rc == 0 and n.value >= last, (m, n.value, last)
        last = n.value


@pytest.mark.gpu
@pytest.mark.parametrize("nq", [129, 1000, 2000])
def test_queries_in_scratch_of_more(L, nq):
    N, d, k = 20_000, 16, 10
    rng = np.random.default_rng(nq)
    X = rng.integers(0, 4, size=(N, d), dtype=np.uint8)
    Q = rng.integers(0, 4, size=(nq, d), dtype=np.uint8)
    have = _query_bytes(L, N, 15_000, d, 3, k)
    ws = torch.empty(have, dtype=torch.uint8, device=DEV)
    Xt, Qt = torch.from_numpy(X).to(DEV), torch.from_numpy(Q).to(DEV)
    ids = torch.empty((nq, k), dtype=torch.int32, device=DEV)
    dist = torch.empty((nq, k), dtype=torch.float32, device=DEV)
    rc = L.ann_knn_query(Xt.data_ptr(), N, Qt.data_ptr(), nq, d, 3, k, ids.data_ptr(),
                         dist.data_ptr(), ws.data_ptr(), have,
                         torch.cuda.current_stream().cuda_stream)
    assert rc == 0, L.ann_last_error()
    torch.cuda.synchronize()
    oi, od = oracle.bruteforce(X, Q, k)
    assert np.array_equal(as_u32(ids), oi)
    assert np.array_equal(dist.cpu().numpy().astype(np.float64), od)
    assert ann.device_status() == 0


# more than 256 centroids: two to four column tiles, split for small launches only
@pytest.mark.gpu
@pytest.mark.parametrize("N,S,C,d", [(10_000, 5_888, 512, 96), (5_000, 2_944, 1024, 128),
                                     (9_000, 700, 300, 20)])
def test_partition_with_a_small_sample(N, S, C, d):
    X = datagen.clustered_u8(N, d, 40, seed=C)
    rng = np.random.default_rng(S)
    sample = np.sort(rng.choice(N, size=S, replace=False)).astype(np.uint32)
    init = X[rng.choice(N, size=C, replace=False)].astype(np.float32)
    t = lambda a: torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).to(DEV)
    cent, mem, off = ann.partition(t(X), C, 2, t(init), t(sample), 2)
    cent_o, _, mem_o, off_o = oracle.partition(X, init, sample, 2, C, 2)
    assert np.array_equal(cent.cpu().numpy().view(np.uint32), cent_o.view(np.uint32))
    assert np.array_equal(off.cpu().numpy(), off_o)
    assert np.array_equal(as_u32(mem), mem_o)
    assert ann.device_status() == 0
