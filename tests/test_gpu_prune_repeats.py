"""ann_prune on lists that hold an id more than once: a neighbour's list counts an id once,
at its first place, as in the oracle.  Compared on the rows whose own list is distinct."""
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


@pytest.mark.parametrize("k,R", [(9, 4), (32, 16), (33, 7), (64, 32), (100, 40), (256, 64)])
def test_repeated_ids_count_once(k, R):
    rng = np.random.default_rng(k)
    mem = np.concatenate([np.arange(700), 1000 + np.arange(300)]).astype(np.uint32)
    off = np.array([0, 700, 1000], dtype=np.int64)
    knn = np.empty((1000, k), dtype=np.uint32)
    for p in range(1000):
        s = int(p >= 700)
        lo, n = (0, 700) if s == 0 else (1000, 300)
        # ids from a small range, so that lists of neighbours meet often
        knn[p] = lo + (p - off[s] + 1 + rng.choice(min(n - 1, k + 8), size=k, replace=False)) % n
        if rng.random() < 0.5:
            knn[p, rng.integers(0, k, size=k // 2)] = knn[p, rng.integers(0, k, size=k // 2)]
    repeats = np.array([len(set(r.tolist())) < k for r in knn])
    assert 100 < repeats.sum() < 900
    d = np.sort(rng.random((1000, k)).astype(np.float32), axis=1)
    t = lambda a: torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).to(DEV)
    ids, dist = ann.prune(t(knn), t(d), t(mem), t(off), R)
    oi, od = oracle.prune(knn, d.astype(np.float64), mem, off, R)
    ok = ~repeats
    assert np.array_equal(as_u32(ids)[ok], oi[ok])
    assert np.array_equal(dist.cpu().numpy()[ok].astype(np.float64), od[ok])
