"""What a user of the library has it do, as timed cases.

Every case goes through the public binding (``paper_1810_07355_gb300.onng`` and
``learned``): single requests and small batches against a serving-sized index,
whole query batches in each stored type, the learned per-query form and the
training of its network, index builds over byte, word-vector and odd-sized
integer data, and exact neighbours of a few queries.

The data are the stand-ins of ``synth.py`` drawn on the GPU from a seed:
  mixture  isotropic Gaussian mixture, 50 centres in [0, 100]^d, sigma 8
  bytes    image descriptors: integers 0-255, about 30 % zeros, 1,000 clusters
  text     unit vectors around 2,000 directions, Zipf(1.1) cluster sizes
  gist     |centre + N(0, 0.1^2)|, 500 centres in [0, 1]^d
"""
from __future__ import annotations

import heapq
import math

import numpy as np
import torch

from paper_1810_07355_gb300 import learned, onng

PRECISIONS = {"fp32": onng.PREC_FP32, "bf16": onng.PREC_BF16, "fp8": onng.PREC_FP8}
WIDTH = {"fp32": 4, "bf16": 2, "fp8": 1}  # bytes of a stored coordinate
CENTRES = {"mixture": 50, "bytes": 1000, "text": 2000, "gist": 500}

# Index settings of the repository's benchmark: k = 100 neighbours, Algorithm 2
# with (20, 60), path adjustment; 10 seeds per query from n_pivot pivots.
GRAPH = dict(graph_k=100, e_o=20, e_i=60)


def listed():
    return [
        # One query against the 10,000-point serving index: the latency of a lone request.
        dict(name="request_1", do="search", data="mixture", n=10_000, d=128, nq=1, k=10, precision="fp32", e_s=20,
             padded=True, eps=0.05, cap=0, n_pivot=1024, visits=160, **GRAPH),
        # A ragged request of the serving trace for 100 neighbours: bfloat16 with the float32
        # rerank, every edge of the CSR lists (the class whose recall needs all edges).
        dict(name="request_137", do="search", data="mixture", n=10_000, d=128, nq=137, k=100, precision="bf16", e_s=0,
             padded=False, eps=0.025, cap=0, n_pivot=1024, visits=200, **GRAPH),
        # The headline batch: 10,000 queries at recall@10 = 0.95 over a million image descriptors,
        # bfloat16 + rerank, expansions capped.
        dict(name="batch_bf16", do="search", data="bytes", n=1_000_000, d=128, nq=10_000, k=10, precision="bf16",
             e_s=20, padded=True, eps=0.07074, cap=389, n_pivot=1024, visits=1900, **GRAPH),
        # The same batch as the paper runs it: float32, no cap.
        dict(name="batch_fp32", do="search", data="bytes", n=1_000_000, d=128, nq=10_000, k=10, precision="fp32",
             e_s=20, padded=True, eps=0.09186, cap=0, n_pivot=1024, visits=1880, **GRAPH),
        # Scene descriptors: long vectors stored as FP8 codes, many pivots.
        dict(name="gist_fp8", do="search", data="gist", n=100_000, d=960, nq=1000, k=10, precision="fp8", e_s=20,
             padded=True, eps=0.01, cap=0, n_pivot=8192, visits=160, **GRAPH),
        # Word vectors: d = 100, concentrated distances, hubs, large candidate sets.
        dict(name="text_fp32", do="search", data="text", n=200_000, d=100, nq=2000, k=10, precision="fp32", e_s=20,
             padded=True, eps=0.085, cap=0, n_pivot=16_384, visits=1600, **GRAPH),
        # The learned form: probe, predictor network, bfloat16 search with per-query (eps, e_s).
        dict(name="learned_bf16", do="learned", data="bytes", n=300_000, d=128, nq=5000, k=10, h=4, n_pivot=1024,
             visits=1600, **GRAPH),
        # Training of the predictor as learned.train calls it: Adam steps of 128 samples.
        dict(name="train", do="train", samples=30_000, batch=128, steps=1000),
        # A million-descriptor index from its vectors: exact kNN graph, degree and path
        # adjustment, padded table.
        dict(name="build_bytes", do="build", data="bytes", n=1_000_000, d=128, e_s=20, **GRAPH),
        # A word-vector index (float values, d = 100).
        dict(name="build_text", do="build", data="text", n=200_000, d=100, e_s=20, **GRAPH),
        # A ragged index of integer descriptors whose dimension is no multiple of 64.
        dict(name="build_odd", do="build", data="bytes", n=30_011, d=100, e_s=20, **GRAPH),
        # Exact neighbours of a handful of queries over the whole base.
        dict(name="exact_50", do="exact", data="bytes", n=1_000_000, d=128, nq=50, k=10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["search", "search", "search", "search", "learned", "train", "build", "build", "exact", "exact"])
    if do == "train":
        return dict(do="train", samples=_log_int(rng, 2000, 60_000), batch=rng.choice([16, 37, 64, 100, 128]),
                    steps=_log_int(rng, 50, 1000))
    if do == "learned":
        return dict(do="learned", data="bytes", n=_log_int(rng, 20_000, 500_000), d=rng.choice([64, 100, 128]),
                    nq=_log_int(rng, 1, 10_000), k=rng.choice([10, 10, 32]), h=rng.choice([4, 8]), n_pivot=1024,
                    visits=1500, **GRAPH)
    data = rng.choice(["mixture", "bytes", "bytes", "text", "gist"])
    most, d = {"mixture": (200_000, rng.choice([32, 64, 96, 128, 256])), "bytes": (600_000, rng.choice([64, 100, 128, 128])),
               "text": (200_000, rng.choice([52, 100, 200])), "gist": (60_000, rng.choice([512, 960]))}[data]
    if data == "bytes" and d == 100:
        most = 60_000
    if do == "exact":
        n = _log_int(rng, 10_000, most)
        return dict(do="exact", data=data, n=n, d=d, nq=_log_int(rng, 1, min(n, 10_000)), k=rng.choice([1, 10, 100]))
    e_o = rng.choice([10, 20])
    graph = dict(graph_k=100, e_o=e_o, e_i=rng.choice([20, 40, 60]))
    if do == "build":
        return dict(do="build", data=data, n=_log_int(rng, 3000, most // 2), d=d, e_s=rng.choice([10, 20]), **graph)
    k = rng.choice([1, 10, 10, 100])
    e_s = rng.choice([10, 20, 20, 40, 0])
    return dict(do="search", data=data, n=_log_int(rng, 5000, most), d=d, nq=_log_int(rng, 1, 10_000 if data == "bytes" else 1000),
                k=k, precision=rng.choice(["fp32", "bf16", "bf16", "fp8"]), e_s=e_s, padded=e_s > 0,
                eps={"mixture": 0.05, "bytes": 0.07, "text": 0.06, "gist": 0.01}[data] * rng.uniform(0.5, 1.2),
                cap=rng.choice([0, 0, 300]), n_pivot=rng.choice([1024, 4096]),
                visits={"mixture": 200, "bytes": 1200, "text": 700, "gist": 160}[data], **graph)


# ----------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _points(data, n, d, g, centres):
    """n rows of the named distribution around the given centres."""
    out = torch.empty((n, d), device="cuda")
    for s in range(0, n, 1 << 17):
        m = min(1 << 17, n - s)
        if data == "text":
            w = 1.0 / torch.arange(1, CENTRES["text"] + 1, device="cuda", dtype=torch.float64) ** 1.1
            comp = torch.multinomial((w / w.sum()).float(), m, replacement=True, generator=g)
            v = centres[comp] + (0.3 / math.sqrt(d)) * torch.randn((m, d), device="cuda", generator=g)
            v /= v.norm(dim=1, keepdim=True)
        else:
            comp = torch.randint(0, len(centres), (m,), device="cuda", generator=g)
            if data == "bytes":
                u = torch.ones((m, d), device="cuda")
                for _ in range(4):  # Gamma(4, 1/4)
                    u *= 1.0 - torch.rand((m, d), device="cuda", generator=g)
                active = torch.rand((m, d), device="cuda", generator=g) < 0.7
                v = (centres[comp] * (-0.25 * u.clamp_min(1e-30).log())).round().clamp_(0, 255) * active
            elif data == "gist":
                v = (centres[comp] + 0.1 * torch.randn((m, d), device="cuda", generator=g)).abs()
            else:
                v = centres[comp] + 8.0 * torch.randn((m, d), device="cuda", generator=g)
        out[s:s + m] = v
    return out


def _base_and_queries(case, seed):
    data, d = case["data"], case["d"]
    g = _gen(seed)
    shape = (CENTRES[data], d)
    if data == "bytes":  # Gamma(2, 20)
        u = 1.0 - torch.rand((2,) + shape, device="cuda", generator=g)
        c = -20.0 * u.clamp_min(1e-30).log().sum(0)
    elif data == "text":
        c = torch.randn(shape, device="cuda", generator=g)
        c /= c.norm(dim=1, keepdim=True)
    else:
        c = torch.rand(shape, device="cuda", generator=g) * (1.0 if data == "gist" else 100.0)
    X = _points(data, case["n"], d, g, c)
    return X, _points(data, case["nq"], d, g, c) if case.get("nq") else None


def _samples(case, seed):
    """Standardised features and (log eps, log e_s) targets of the predictor's training."""
    g = _gen(seed)
    X = torch.randn((case["samples"], 16), device="cuda", generator=g)
    w = 0.3 * torch.randn((16, 2), device="cuda", generator=g)
    T = (X @ w).tanh() + 0.3 * torch.randn((case["samples"], 2), device="cuda", generator=g)
    return X, T + torch.tensor([-2.6, 2.7], device="cuda")


def prepare(case, seed):
    if case["do"] == "train":
        X, T = _samples(case, seed)
        return dict(case=case, X=X, T=T, P0=onng.mlp_init(seed))
    X, Q = _base_and_queries(case, seed)
    state = dict(case=case, X=X, Q=Q)
    if case["do"] in ("search", "learned"):
        index = onng.build_index(X, case["graph_k"], case["e_o"], case["e_i"])
        if case["do"] == "learned":
            index.with_adjacency(20).with_bf16()
            P = onng.mlp_init(seed)  # a network whose outputs lie around eps 0.07 and e_s 16
            P[-130:-2] *= 0.02
            P[-2:] = torch.tensor([math.log(0.07 + learned.EPS_FLOOR), math.log(16.0)], device="cuda")
            state["predictor"] = learned.Predictor(P, h=case["h"])
        else:
            if case["padded"]:
                index.with_adjacency(case["e_s"])
            if case["precision"] == "bf16":
                index.with_bf16()
            elif case["precision"] == "fp8":
                index.with_fp8()
            state["workspace"] = onng.SearchWorkspace()
        state["index"] = index
    if case["do"] == "build":  # the program keeps its graph in arrays that hold any index of these settings
        room = case["n"] * (case["e_o"] + case["e_i"])
        state["col"] = torch.full((room,), -1, dtype=torch.int32, device="cuda")
        state["length"] = torch.full((room,), math.inf, device="cuda")
    return state


# ----------------------------------------------------------------------------- one pass

def run(state):
    case, do = state["case"], state["case"]["do"]
    if do == "train":
        P = state["P0"].clone()
        M, V = torch.zeros_like(P), torch.zeros_like(P)
        onng.mlp_train(P, M, V, state["X"], state["T"], case["steps"], case["batch"], 2e-3)
        return dict(P=P, M=M, V=V)
    if do == "exact":
        ids, dist = onng.knn(state["X"], state["Q"], case["k"])
        return dict(ids=ids, dist=dist)
    if do == "build":
        index = onng.build_index(state["X"], case["graph_k"], case["e_o"], case["e_i"]).with_adjacency(case["e_s"])
        state["col"][:index.col.numel()].copy_(index.col)
        state["length"][:index.col.numel()].copy_(index.length)
        return dict(row_ptr=index.row_ptr, col=state["col"], length=state["length"], adj=index.adj)
    index, Q = state["index"], state["Q"]
    seeds = onng.seeds_pivot(index.X, Q, case["n_pivot"], 10)
    if do == "learned":
        ids, dist, st, eps_q, es_q = learned.learned_search(state["predictor"], index, Q, case["k"], seeds, 0.95,
                                                            k_rerank=max(20, case["k"]))
        return dict(ids=ids, dist=dist, stats=st, eps=eps_q, es=es_q)
    rerank = 0 if case["precision"] == "fp32" else max(20, case["k"])
    ids, dist, st = onng.search(index, Q, case["k"], case["e_s"], case["eps"], seeds,
                                precision=PRECISIONS[case["precision"]], k_rerank=rerank, max_expansions=case["cap"],
                                workspace=state["workspace"])
    return dict(ids=ids, dist=dist, stats=st, seeds=seeds)


# ----------------------------------------------------------------------------- what a pass cannot do without

def work(case):
    """Inputs read once, outputs written once, and the arithmetic of the method.  A search
    reads one vector per distance computation (`visits`: about how many a query takes on
    such an index); a build is the distance sweep and the index it writes (about 17 edges
    a node)."""
    if case["do"] == "train":
        return {"bytes": case["samples"] * 72 + 6 * 5378 * 4, "flops": case["steps"] * case["batch"] * 6 * 5248}
    n, d, nq = case["n"], case["d"], case.get("nq", 0)
    if case["do"] == "exact":
        return {"bytes": (n + nq) * d * 4 + nq * case["k"] * 8, "flops": 2 * n * nq * d}
    if case["do"] == "build":
        return {"bytes": n * (4 * d + 17 * 8 + 8 + 4 * case["e_s"]), "flops": 2 * n * n * d}
    width = WIDTH[case.get("precision", "bf16")]
    pivots = min(case["n_pivot"], n)
    per_query = case["visits"] * d * width + case["visits"] / 13 * 20 * 4 + 4 * d + 8 * case["k"] + 16 + 40
    return {"bytes": int(nq * per_query + pivots * d * 4), "flops": int(nq * (case["visits"] + pivots) * d * 3)}


# ----------------------------------------------------------------------------- the same in 64 bits

def _exact_knn(X, Q, k, self_join):
    """(ids, lengths) of the k nearest by (distance, id) in float64."""
    X, ids, out = X.double(), [], []
    xn = (X * X).sum(1)
    step = max(1, int(6e7 // X.shape[0]))
    for s in range(0, Q.shape[0], step):
        q = Q[s:s + step].double()
        d2 = (q * q).sum(1)[:, None] + xn[None, :] - 2.0 * (q @ X.T)
        if self_join:
            r = torch.arange(len(q), device="cuda")
            d2[r, r + s] = math.inf
        v, i = torch.sort(d2, dim=1, stable=True)
        ids.append(i[:, :k].clone())
        out.append(v[:, :k].clamp_min(0).sqrt())
    return torch.cat(ids), torch.cat(out)


def _exact_graph(X, case):
    """Row pointers, columns and lengths of the degree- and path-adjusted graph in float64."""
    n, k = X.shape[0], case["graph_k"]
    nbr, ln = _exact_knn(X, X, k, True)
    rows = torch.arange(n, device="cuda")[:, None].expand(n, k)
    e_o, e_i = case["e_o"], case["e_i"]
    src = torch.cat([rows[:, :e_o].reshape(-1), nbr[:, :e_i].reshape(-1)])
    dst = torch.cat([nbr[:, :e_o].reshape(-1), rows[:, :e_i].reshape(-1)])
    val = torch.cat([ln[:, :e_o].reshape(-1), ln[:, :e_i].reshape(-1)])
    key, inv = torch.unique(src * n + dst, return_inverse=True)
    length = torch.empty(len(key), dtype=torch.float64, device="cuda")
    length[inv] = val  # the same pair has the same length in both directions
    o = torch.sort(length, stable=True).indices  # rows by (length, id): the keys are in id order
    key, length = key[o], length[o]
    o = torch.sort(key // n, stable=True).indices
    key, length = key[o], length[o]
    src, dst = key // n, key % n
    ptr = torch.searchsorted(src.contiguous(), torch.arange(n + 1, device="cuda"))
    skey, order = torch.sort(key)
    slen, keep = length[order], torch.ones(len(key), dtype=torch.bool, device="cuda")
    deg = ptr[1:] - ptr[:-1]
    for s in range(0, len(key), 1 << 19):  # all i -> m -> j: drop (i, j) where both hops are shorter
        m = dst[s:s + (1 << 19)]
        reps = deg[m]
        first = torch.repeat_interleave(torch.arange(len(m), device="cuda"), reps)
        e2 = torch.arange(len(first), device="cuda") - torch.repeat_interleave(reps.cumsum(0) - reps, reps) + ptr[m][first]
        want = src[s + first] * n + dst[e2]
        at = torch.searchsorted(skey, want).clamp_max(len(skey) - 1)
        hit = (skey[at] == want) & (length[s + first] < slen[at]) & (length[e2] < slen[at])
        keep[order[at[hit]]] = False
    ptr = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), keep.long().cumsum(0)])[ptr]
    return ptr, dst[keep], length[keep]


def _exact_search(ptr, col, X, q, seeds, case, kept, stored):
    """Algorithm 1 for one query: ids, distances and counts."""
    def dist(ids):
        t = stored[ids] - q
        return np.sqrt((t * t).sum(1))
    seen, r, bound = set(seeds.tolist()), math.inf, math.inf
    S = sorted(zip(dist(seeds).tolist(), seeds.tolist()))
    R = [(-a, -b) for a, b in S[:kept]]
    heapq.heapify(R)
    computed, expanded, scanned = len(S), 0, 0
    while S and S[0][0] <= bound:
        if case["cap"] and expanded >= case["cap"]:
            break
        node = heapq.heappop(S)[1]
        row = col[ptr[node]:ptr[node + 1]]
        row = row[:case["e_s"]] if case["e_s"] > 0 else row
        expanded, scanned = expanded + 1, scanned + len(row)
        new = [i for i in row.tolist() if i not in seen]
        if not new:
            continue
        seen.update(new)
        computed += len(new)
        for a, b in zip(dist(np.array(new)).tolist(), new):
            if a <= bound:
                heapq.heappush(S, (a, b))
            if a <= r:
                heapq.heappush(R, (-a, -b))
                if len(R) > kept:
                    heapq.heappop(R)
                if len(R) == kept:
                    r = -R[0][0]
                    bound = r * (1.0 + case["eps"])
    ids = np.array([-b for _, b in R])
    t = X[ids] - q  # the float32 rerank of a reduced form; the same values otherwise
    got = sorted(zip(np.sqrt((t * t).sum(1)).tolist(), ids.tolist()))[:case["k"]]
    return got, (computed, expanded, scanned, 0)


def _exact_train(case, seed):
    X, T = (v.double() for v in _samples(case, seed))
    P = onng.mlp_init(seed).double()
    M, V = torch.zeros_like(P), torch.zeros_like(P)
    cut = [16 * 64, 64, 64 * 64, 64, 2 * 64, 2]
    N, B = case["samples"], case["batch"]
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    for step in range(case["steps"]):
        rows = (torch.arange(B, device="cuda") + step * B) % N
        x, t = X[rows], T[rows]
        w1, c1, w2, c2, w3, c3 = torch.split(P, cut)
        w1, w2, w3 = w1.view(64, 16), w2.view(64, 64), w3.view(2, 64)
        h1 = (x @ w1.T + c1).clamp_min(0)
        h2 = (h1 @ w2.T + c2).clamp_min(0)
        dy = (h2 @ w3.T + c3 - t) / B
        d2 = (dy @ w3) * (h2 > 0)
        d1 = (d2 @ w2) * (h1 > 0)
        G = torch.cat([(d1.T @ x).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), (dy.T @ h2).reshape(-1), dy.sum(0)])
        M = b1 * M + (1 - b1) * G
        V = b2 * V + (1 - b2) * G * G
        P = P - float(np.float32(2e-3)) * (M / (1 - b1 ** (step + 1))) / ((V / (1 - b2 ** (step + 1))).sqrt() + float(np.float32(1e-8)))
    return dict(P=P, M=M, V=V)


def exact(case, seed):
    if case["do"] == "train":
        return _exact_train(case, seed)
    if case["do"] == "learned":
        return None  # starts from features of a capped search, which have no value but the search's own
    X, Q = _base_and_queries(case, seed)
    n = case["n"]
    if case["do"] == "exact":
        if n * case["nq"] > 3e8:
            return None
        ids, dist = _exact_knn(X, Q, case["k"], False)
        return dict(ids=ids, dist=dist)
    if n > 32_000:
        return None  # the 64-bit graph would take too long
    if case["do"] == "build":
        ptr, col, length = _exact_graph(X, case)
        pos = torch.arange(case["e_s"], device="cuda")[None, :] + ptr[:-1, None]
        adj = torch.where(pos < ptr[1:, None], col[pos.clamp_max(len(col) - 1)], -1)
        room = n * (case["e_o"] + case["e_i"]) - len(col)
        return dict(row_ptr=ptr, col=torch.nn.functional.pad(col, (0, room), value=-1),
                    length=torch.nn.functional.pad(length, (0, room), value=math.inf), adj=adj)
    if case["precision"] == "fp8" or case["nq"] * case["k"] > 20_000:
        return None  # FP8 codes are a rounding of their own
    P = min(case["n_pivot"], n)
    pivots = torch.arange(P, device="cuda") * n // P
    seeds = pivots[_exact_knn(X[pivots], Q, 10, False)[0]]
    ptr, col, _ = (v.cpu().numpy() for v in _exact_graph(X, case))
    x, q, s = X.double().cpu().numpy(), Q.double().cpu().numpy(), seeds.cpu().numpy()
    stored = X.bfloat16().double().cpu().numpy() if case["precision"] == "bf16" else x
    kept = case["k"] if case["precision"] == "fp32" else max(20, case["k"])
    ids, dist = np.full((case["nq"], case["k"]), -1), np.full((case["nq"], case["k"]), math.inf)
    stats = np.zeros((case["nq"], 4), dtype=np.int64)
    for i in range(case["nq"]):
        got, stats[i] = _exact_search(ptr, col, x, q[i], s[i], case, kept, stored)
        dist[i, :len(got)] = [a for a, _ in got]
        ids[i, :len(got)] = [b for _, b in got]
    return dict(ids=ids, dist=dist, stats=stats, seeds=seeds)
