"""The calls that a user of this framework makes, at the sizes they come in.

A case is a dict: the kind of call, the shape of the vectors (N, d, dtype and the
distribution they are drawn from) and the parameters of the build or the query.

  build          ann.build_index: partition, per-shard kNN, prune, merge (with "reverse",
                 the reverse edges added to the merged graph as well)
  shards         ann.build_from_shards: the same over a partition made elsewhere
  selective      ann.build_index with the selective replication of the partition
  learned_train  ann.learned_train: the projection network of the learned form
  learned_knn    ann.learned_embed and the learned form of ann.shard_knn
  query          ann.knn_query: exact neighbours of queries (ground truth)
  search         ann.search_entries / ann.search on a finished graph

Vectors are drawn on the device from the seed; the distributions are those of
paper_2605_10135_gb300.datagen (clustered integers, anisotropic mixtures on the unit
sphere, power-law spectra), which is what the benchmark's workloads consist of.
"""
from __future__ import annotations

import math

import torch

from paper_2605_10135_gb300 import ann

DEV = "cuda"
DTYPES = {"u8": torch.uint8, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BYTES = {"u8": 1, "f32": 4, "f16": 2, "bf16": 2}
PRECISION = {"exact": ann.EXACT, "bf16": ann.BF16_RERANK, "fp8": ann.FP8_RERANK,
             "f16": ann.F16_RERANK}
LEARNED_STEPS, LEARNED_BATCH, HIDDEN, OUT = 300, 512, 256, 32


# ---- the cases --------------------------------------------------------------------
def listed():
    return [
        # A small collection (the repository's small float workload): the whole build is
        # a few hundred short kernels, so launches and latency are what a user waits for.
        dict(name="build_gauss10k_f32", kind="build", data="gauss", N=10_000, d=64, dtype="f32",
             C=4, r=2, k=32, R=16, precision="exact", reverse=False),
        # An odd collection: rows of 100 bytes, sizes that are no multiple of anything,
        # three replicas, BF16 vectors, and reverse edges on the merged graph.
        dict(name="build_ragged_bf16", kind="build", data="embed", N=77_777, d=50, dtype="bf16",
             C=11, r=3, k=48, R=20, precision="exact", reverse=True),
        # The integer workload of the paper's shape (uint8 descriptors of 128 dimensions).
        dict(name="build_sift1m_u8", kind="build", data="sift", N=1_000_000, d=128, dtype="u8",
             C=16, r=2, k=64, R=32, precision="exact", reverse=False),
        # The benchmark's default workload, the largest build.
        dict(name="build_deep10m_f32", kind="build", data="deep", N=10_000_000, d=96, dtype="f32",
             C=64, r=2, k=64, R=32, precision="exact", reverse=False),
        # Selective replication (part of the vectors in one shard only) with the FP16
        # screening form.
        dict(name="selective_deep2m_f16form", kind="selective", data="deep", N=2_000_000, d=96,
             dtype="f32", C=64, r=2, k=64, R=32, precision="f16", epsilon=1.1, capacity=0),
        # Wide float rows in given shards of very uneven size (log-uniform).
        dict(name="shards_laion250k_f32", kind="shards", data="laion", N=250_000, d=768,
             dtype="f32", C=32, r=2, k=32, R=32, precision="exact"),
        # Half-precision embeddings of 1024 dimensions, exact form.
        dict(name="build_embed200k_f16", kind="build", data="embed", N=200_000, d=1024, dtype="f16",
             C=16, r=2, k=64, R=32, precision="exact", reverse=False),
        # The learned form: its training (forward, backward, Adam) on a 1% sample ...
        dict(name="learned_train_200k_f16", kind="learned_train", data="embed", N=200_000, d=1024,
             dtype="f16", S=2_000),
        # ... and the shard lists that a network proposes: 256 candidates a row.  (The
        # parameters are He-initialised; the time does not depend on how good they are.)
        dict(name="learned_knn_200k_f16", kind="learned_knn", data="embed", N=200_000, d=1024,
             dtype="f16", C=8, r=2, k=64, rerank_k=256),
        # Ground truth of a thousand held-out queries against the integer collection.
        dict(name="query_1k_sift1m_u8", kind="query", data="sift", N=1_000_000, d=128, dtype="u8",
             nq=1_000, k=10),
        # Serving: a large batch of queries on a finished graph, from sampled entries.
        dict(name="search_10k_sift400k_u8", kind="search", data="sift", N=400_000, d=128,
             dtype="u8", nq=10_000, Ls=64, topk=10, entries=1024),
        # Serving one query: nothing but latency.
        dict(name="search_one_deep100k_f32", kind="search", data="deep", N=100_000, d=96,
             dtype="f32", nq=1, Ls=64, topk=10, entries=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_DATA = {  # distribution -> (element types, dimensions) it comes with
    "gauss": (("f32", "bf16", "f16"), (16, 64, 100, 33)),
    "sift": (("u8",), (128, 128, 96, 100, 200)),
    "deep": (("f32", "f32", "bf16"), (96, 96, 100, 128, 75)),
    "laion": (("f32", "f16"), (768, 512, 300)),
    "embed": (("f16", "bf16"), (1024, 512, 256, 50)),
}


def draw(rng):
    kind = rng.choice(["build", "build", "build", "build", "shards", "selective", "learned_train",
                       "learned_knn", "query", "query", "search", "search"])
    if kind in ("learned_train", "learned_knn"):
        data = rng.choice(["embed", "laion"])
    elif kind == "shards":
        data = rng.choice(["laion", "embed", "deep", "sift"])
    elif kind == "selective":
        data = rng.choice(["deep", "sift", "gauss"])
    else:
        data = rng.choice(["gauss", "sift", "sift", "deep", "deep", "laion", "embed"])
    dts, dims = _DATA[data]
    dtype, d = rng.choice(dts), rng.choice(dims)
    # rows x columns x dimensions of a build grow with N^2 d: wide rows stay smaller
    most = 4_000_000 if d <= 128 else 400_000 if d <= 300 else 250_000
    c = dict(kind=kind, data=data, d=d, dtype=dtype)
    if kind in ("build", "shards", "selective"):
        c["N"] = N = _log(rng, 4_000, most)
        c["C"] = C = max(2, min(64, _log(rng, 0.5, 2.0) * max(1, round(math.sqrt(N) / 50))))
        c["r"] = 2 if kind != "build" else rng.choice([1, 2, 2, 2, 3]) if C >= 3 else 1
        c["k"] = k = rng.choice([16, 32, 48, 64, 64])
        c["R"] = rng.choice([k // 2, k // 2, k // 2, 20])
        c["R"] = min(c["R"], k)
        c["precision"] = "exact"
        if dtype == "f32" and rng.random() < 0.25:
            c["precision"] = rng.choice(["f16", "bf16", "f16"])
        if kind == "build":
            c["reverse"] = rng.random() < 0.3
        if kind == "selective":
            c["epsilon"] = rng.choice([1.1, 1.2, 1.5])
            c["capacity"] = int(1.2 * 2 * N / C) if N <= 300_000 and rng.random() < 0.3 else 0
    elif kind == "learned_train":
        c["N"] = _log(rng, 20_000, 250_000)
        c["S"] = max(256, c["N"] // 100)
    elif kind == "learned_knn":
        c["N"] = N = _log(rng, 10_000, 250_000)
        c["C"], c["r"], c["k"] = rng.choice([4, 8, 16]), 2, rng.choice([32, 64])
        c["rerank_k"] = rng.choice([128, 256])
    elif kind == "query":
        c["N"] = _log(rng, 10_000, 2_000_000 if d <= 128 else 250_000)
        c["nq"] = _log(rng, 1, 10_000)
        c["k"] = rng.choice([10, 10, 10, 100, 1])
    else:
        c["N"] = _log(rng, 5_000, 400_000 if d <= 128 else 100_000)
        c["nq"] = _log(rng, 1, 10_000)
        c["Ls"], c["topk"] = rng.choice([32, 64, 64, 100, 128]), 10
        c["entries"] = rng.choice([0, 256, 1024])
    return c


# ---- inputs -----------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1_000_003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32)


def _rotation(g, d):
    q, r = torch.linalg.qr(torch.randn(d, d, generator=g, device=DEV, dtype=torch.float64))
    return (q * torch.sign(torch.diagonal(r))[None, :]).float()


def _components(case):
    return {"gauss": 16, "sift": 256, "deep": 1024, "laion": 1,
            "embed": max(16, min(4096, case["N"] // 1000))}[case["data"]]


def _vectors(case, seed, n, salt=0):
    """n rows of the case's distribution; the distribution itself (centres, rotations)
    depends on the seed alone, the draw of the rows on (seed, salt)."""
    d, data, dt = case["d"], case["data"], DTYPES[case["dtype"]]
    g, h = _gen(seed, 11), _gen(seed, 1000 + salt)
    out = torch.empty(n, d, dtype=dt, device=DEV)
    nc = _components(case)
    step = 1 << 20
    if data in ("deep", "embed"):
        sd = 1.0 / torch.arange(1, d + 1, device=DEV, dtype=torch.float64)
        sd = torch.sqrt(sd * (0.25 / sd.sum())).float()
        centres = _normal(g, nc, d)
        rots = [_rotation(g, d) for _ in range(4 if d > 256 else 16)]
    elif data == "laion":
        sd = torch.arange(1, d + 1, device=DEV, dtype=torch.float32) ** -0.4
        rot = _rotation(g, d)
    elif data == "sift":
        centres = torch.rand(nc, d, generator=g, device=DEV) * 192.0 + 32.0
    else:
        centres = _normal(g, nc, d) * 2.0
    for a in range(0, n, step):
        b = min(n, a + step)
        z = _normal(h, b - a, d)
        if data == "laion":
            out[a:b] = ((z * sd) @ rot.T).to(dt)
            continue
        lab = torch.randint(nc, (b - a,), generator=h, device=DEV)
        if data == "sift":
            out[a:b] = torch.clamp(torch.round(centres[lab] + 20.0 * z), 0, 255).to(dt)
        elif data == "gauss":
            out[a:b] = (centres[lab] + z).to(dt)
        else:
            z *= sd
            v = centres[lab]
            rid = lab % len(rots)
            for q, rot in enumerate(rots):
                m = (rid == q).nonzero(as_tuple=True)[0]
                v[m] += z[m] @ rot.T
            if data == "deep":
                v /= v.norm(dim=1, keepdim=True)
            out[a:b] = v.to(dt)
    return out


def _kmeans_inputs(X, case, seed):
    """The sample rows and the initial centroids (the repository's recipe)."""
    N, C = X.shape[0], case["C"]
    g = _gen(seed, 12)
    S = min(N, max(256 * C, N // 100))
    sample = torch.sort(torch.randperm(N, generator=g, device=DEV)[:S])[0]
    rows = sample[torch.randperm(S, generator=g, device=DEV)[:C]]
    return sample.to(torch.int32), X[rows].float()


def _given_shards(case, seed):
    """C shards of log-uniform size, every vector in two of them: each half of the
    shards splits all vectors."""
    N, C = case["N"], case["C"]
    g = _gen(seed, 13)
    members, sizes = [], []
    for half in (C // 2, C - C // 2):
        raw = torch.exp(torch.rand(half, generator=g, device=DEV, dtype=torch.float64)
                        * math.log(80.0))
        cut = torch.round(torch.cumsum(raw, 0) / raw.sum() * N).long().tolist()
        perm = torch.randperm(N, generator=g, device=DEV)
        a = 0
        for b in cut:
            members.append(torch.sort(perm[a:b])[0].to(torch.int32))
            sizes.append(b - a)
            a = b
    off = [0]
    for n in sizes:
        off.append(off[-1] + n)
    return torch.cat(members), torch.tensor(off, dtype=torch.int64, device=DEV)


def _params(d, seed):
    """The parameters of a projection network (He-initialised rows, small biases)."""
    g = _gen(seed, 14)
    return torch.cat([(_normal(g, HIDDEN, d) * math.sqrt(2.0 / d)).reshape(-1),
                      0.01 * _normal(g, HIDDEN),
                      (_normal(g, OUT, HIDDEN) * math.sqrt(1.0 / HIDDEN)).reshape(-1),
                      0.01 * _normal(g, OUT)])


def _config(case):
    sel = None
    if case["kind"] == "selective":
        sel = ann.SelectiveConfig(epsilon=case["epsilon"], capacity=case["capacity"], cand=8)
    return ann.BuildConfig(C=case["C"], r=case["r"], k=case["k"], R=case["R"],
                           precision=PRECISION[case["precision"]], selective=sel)


def prepare(case, seed):
    kind = case["kind"]
    X = _vectors(case, seed, case["N"])
    s = dict(case=case, X=X)
    if kind in ("build", "selective"):
        s["cfg"] = _config(case)
        s["sample"], s["init"] = _kmeans_inputs(X, case, seed)
    elif kind == "shards":
        s["cfg"] = _config(case)
        s["members"], s["offsets"] = _given_shards(case, seed)
    elif kind == "learned_train":
        g = _gen(seed, 15)
        s["sample"] = torch.sort(torch.randperm(case["N"], generator=g, device=DEV)
                                 [:case["S"]])[0].to(torch.int32)
        s["draws"] = torch.randint(-2**31, 2**31, (LEARNED_STEPS, LEARNED_BATCH, 3), generator=g,
                                   device=DEV, dtype=torch.int64).to(torch.int32)
        s["params0"] = _params(case["d"], seed)
    elif kind == "learned_knn":
        sample, init = _kmeans_inputs(X, case, seed)
        _, s["members"], s["offsets"] = ann.partition(X, case["C"], case["r"], init, sample, 4)
        s["params"] = _params(case["d"], seed)
    elif kind == "query":
        s["Q"] = _vectors(case, seed, case["nq"], salt=1)
    else:
        s["Q"] = _vectors(case, seed, case["nq"], salt=1)
        c = dict(case, C=max(2, round(math.sqrt(case["N"]) / 100)))
        sample, init = _kmeans_inputs(X, c, seed)
        out = ann.build_index(X, ann.BuildConfig(C=c["C"], r=2, k=64, R=32, iters=4), init, sample)
        s["graph"], s["degree"] = out["graph"], out["degree"]
        if case["entries"]:
            g = _gen(seed, 16)
            s["entries"] = torch.randperm(case["N"], generator=g,
                                          device=DEV)[:case["entries"]].to(torch.int32)
        else:
            s["entry"] = int(ann.medoid(X).item())
        del out
    torch.cuda.synchronize()
    return s


_KEYS = ("centroids", "members", "offsets", "knn_id", "knn_d", "pr_id", "pr_d", "graph", "gdist",
         "degree")


def run(s):
    case, X = s["case"], s["X"]
    kind = case["kind"]
    if kind == "selective":  # the shard rows' number varies with the data: the merged graph
        out = ann.build_index(X, s["cfg"], s["init"], s["sample"])
        return {n: out[n] for n in ("centroids", "offsets", "graph", "gdist", "degree",
                                    "selective_stats")}
    if kind == "build":
        out = ann.build_index(X, s["cfg"], s["init"], s["sample"])
        res = {n: out[n] for n in _KEYS}
        if case.get("reverse"):
            res["rev_graph"], res["rev_dist"], res["rev_degree"] = ann.merge_reverse(
                out["graph"], out["gdist"], out["degree"])
        return res
    if kind == "shards":
        out = ann.build_from_shards(X, s["members"], s["offsets"], s["cfg"])
        return {n: out[n] for n in ("knn_id", "knn_d", "pr_id", "pr_d", "graph", "gdist", "degree")}
    if kind == "learned_train":
        params = s["params0"].clone()  # trained in place
        losses, est = ann.learned_train(X, s["sample"], s["draws"], params)
        return dict(params=params, losses=losses, recall=est)
    if kind == "learned_knn":
        E = ann.learned_embed(X, s["params"])  # kept for embedding-space queries
        ids, dist = ann.shard_knn(X, s["members"], s["offsets"], case["k"], ann.LEARNED,
                                  case["rerank_k"], s["params"])
        return dict(E=E, knn_id=ids, knn_d=dist)
    if kind == "query":
        ids, dist = ann.knn_query(X, s["Q"], case["k"])
        return dict(ids=ids, dist=dist)
    if case["entries"]:
        ids, cnt = ann.search_entries(s["graph"], s["degree"], X, s["Q"], s["entries"], case["Ls"],
                                      case["topk"])
    else:
        ids, cnt = ann.search(s["graph"], s["degree"], X, s["Q"], s["entry"], case["Ls"],
                              case["topk"])
    return dict(ids=ids, count=cnt)


# ---- what a pass cannot do without --------------------------------------------------
def _near(case, n):
    """Columns that every row of n candidates has to be compared with: those of its own
    mixture component (clustered data: the triangle inequality can rule out the
    others), all of them where the data has no clusters or the rows are wide."""
    if case["data"] == "laion" or case["d"] > 200:
        return n
    return min(n, case["N"] / _components(case))


def work(case):
    N, d, e, kind = case["N"], case["d"], BYTES[case["dtype"]], case["kind"]
    if kind in ("build", "selective", "shards"):
        rows, k, R = N * case["r"], case["k"], case["R"]
        if kind == "selective":
            rows = N * 1.5
        outs = rows * (4 + 8 * k + 8 * R) + N * (8 * R + 4)
        flops = 2.0 * d * rows * _near(case, rows / case["C"])
        if kind != "shards":
            flops += 2.0 * d * N * case["C"]
        if case.get("reverse"):
            outs += N * (8 * R + 4)
        return dict(bytes=float(N * d * e + outs), flops=float(flops))
    P = HIDDEN * d + HIDDEN + OUT * HIDDEN + OUT
    mlp = 2.0 * (HIDDEN * d + OUT * HIDDEN)
    if kind == "learned_train":
        train = LEARNED_STEPS * 3 * LEARNED_BATCH * mlp * 3.0
        flops = train + 2.0 * d * case["S"] * N + N * mlp + 2.0 * OUT * case["S"] * N
        return dict(bytes=float(N * d * e + 8 * P), flops=flops)
    if kind == "learned_knn":
        rows, k = N * case["r"], case["k"]
        flops = N * mlp + 2.0 * OUT * rows * rows / case["C"] + 2.0 * d * rows * case["rerank_k"]
        return dict(bytes=float(N * d * e + 4 * P + N * OUT * 4 + rows * (4 + 8 * k)), flops=flops)
    if kind == "query":
        return dict(bytes=float(N * d * e + case["nq"] * (d * e + 8 * case["k"])),
                    flops=2.0 * d * case["nq"] * N)
    # a search has to measure the list it returns from and the neighbours of that list
    seen = case["Ls"] * 8 + case["entries"]
    return dict(bytes=float(case["nq"] * (seen * d * e + case["Ls"] * 32 * 4)),
                flops=2.0 * d * case["nq"] * seen)


# ---- 64-bit values --------------------------------------------------------------------
def _d32(X, cent):
    """Squared distances as the partition decides on them: FP32, index order, unfused."""
    s = torch.zeros(X.shape[0], cent.shape[0], device=X.device, dtype=torch.float32)
    for t in range(X.shape[1]):
        df = X[:, t, None] - cent[None, :, t]
        s = s + df * df
    return s


def _exact_partition(X, case, init, sample, iters=10):
    """Lloyd's iterations with 64-bit means, then each vector's r nearest centroids."""
    Xf = X.float()
    S = Xf[sample.long()]
    S64 = S.double()
    C = case["C"]
    cent = init.double()
    for _ in range(iters):
        lab = torch.argmin(_d32(S, cent.float()), 1)
        n = torch.bincount(lab, minlength=C)
        sums = torch.zeros(C, X.shape[1], device=DEV, dtype=torch.float64)
        sums.index_add_(0, lab, S64)
        mean = sums / n.clamp(min=1)[:, None]
        cent = torch.where((n > 0)[:, None], mean, cent.float().double())
    near = []
    for a in range(0, X.shape[0], 1 << 17):
        near.append(torch.sort(_d32(Xf[a:a + (1 << 17)], cent.float()), dim=1, stable=True)[1]
                    [:, :case["r"]])
    near = torch.cat(near)
    members, off = [], [0]
    for c in range(C):
        m = (near == c).any(1).nonzero(as_tuple=True)[0]
        members.append(m)
        off.append(off[-1] + m.numel())
    return cent, torch.cat(members), off


def _exact_lists(Q, X, k, skip=None):
    """The k smallest squared distances of each row of Q to the rows of X in 64 bits,
    ascending (skip[i]: the row of X that row i leaves out); 32-bit products screen
    k + 48 candidates."""
    n = X.shape[0]
    Xf = X.float()
    nx = (Xf * Xf).sum(1)
    X64 = X.double() if X.numel() <= (1 << 28) else None
    out = torch.full((Q.shape[0], k), math.inf, device=DEV, dtype=torch.float64)
    w = min(n, k + 48)
    ch = max(1, min((1 << 28) // max(n, 1), (1 << 28) // (w * X.shape[1])))
    for a in range(0, Q.shape[0], ch):
        q = Q[a:a + ch]
        key = torch.addmm(nx[None, :].expand(q.shape[0], n), q.float(), Xf.T, alpha=-2.0)
        if skip is not None:
            key[torch.arange(q.shape[0], device=DEV), skip[a:a + ch]] = math.inf
        val, idx = torch.topk(key, w, 1, largest=False, sorted=False)
        c = X64[idx] if X64 is not None else X[idx].double()
        d64 = (c - q.double()[:, None, :]).square_().sum(2)
        d64[torch.isinf(val)] = math.inf
        d64 = torch.sort(d64, 1)[0][:, :k]
        out[a:a + ch, :d64.shape[1]] = d64
    return out


def _exact_shards(X, members, off, k):
    return torch.cat([_exact_lists(X[members[a:b].long()], X[members[a:b].long()], k,
                                   torch.arange(b - a, device=DEV))
                      for a, b in zip(off[:-1], off[1:])])


def exact(case, seed):
    kind, N = case["kind"], case["N"]
    if kind in ("search", "selective") or case.get("precision", "exact") != "exact":
        return None  # integers, or lists whose members an approximate screen decides
    if kind == "learned_train":
        return None  # 300 Adam steps: parameters with vanishing gradients follow the rounding
    if kind in ("build", "shards") and 2.0 * N * N * 2 / case["C"] > 6e10:
        return None  # minutes of 64-bit distances
    s = prepare(case, seed)
    X = s["X"]
    if kind == "build":
        cent, members, off = _exact_partition(X, case, s["init"], s["sample"])
        res = {n: None for n in _KEYS}
        res["centroids"], res["knn_d"] = cent, _exact_shards(X, members, off, case["k"])
        if case.get("reverse"):
            res.update(rev_graph=None, rev_dist=None, rev_degree=None)
        return res
    if kind == "shards":
        res = dict.fromkeys(("knn_id", "knn_d", "pr_id", "pr_d", "graph", "gdist", "degree"))
        res["knn_d"] = _exact_shards(X, s["members"], s["offsets"].tolist(), case["k"])
        return res
    if kind == "query":
        return dict(ids=None, dist=_exact_lists(s["Q"], X, case["k"]))
    p, d = s["params"].double(), case["d"]
    o1, o2, o3 = HIDDEN * d, HIDDEN * d + HIDDEN, HIDDEN * d + HIDDEN + OUT * HIDDEN
    scale = float(X.double().abs().max())
    E = torch.empty(N, OUT, device=DEV, dtype=torch.float64)
    for a in range(0, N, 1 << 16):
        h = (X[a:a + (1 << 16)].double() / scale @ p[:o1].view(HIDDEN, d).T + p[o1:o2]).clamp(min=0)
        E[a:a + (1 << 16)] = h @ p[o2:o3].view(OUT, HIDDEN).T + p[o3:]
    return dict(E=E, knn_id=None, knn_d=None)
