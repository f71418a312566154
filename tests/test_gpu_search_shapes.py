"""The search at the shapes where its gathers, its visited table and its candidate levels
change form: results and counts equal Algorithm 1's on integer data."""
import numpy as np
import pytest

import oracle
from paper_1810_07355_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _compare(X, Q, g, seeds, k, e_s, eps, padded, prec, cap=0):
    from paper_1810_07355_gb300 import onng
    idx = onng.Index(_dev(g[0].astype(np.int64)), _dev(g[1].astype(np.int32)), _dev(X))
    if padded:
        idx.with_adjacency(padded)
    ids, dist, st = onng.search(idx, _dev(Q), k, e_s, eps, _dev(seeds), precision=prec, k_rerank=k, max_expansions=cap)
    o_ids, o_dist, o_st = oracle.search(g[0], g[1], X, Q, k, e_s, np.float32(eps), seeds, max_exp=cap)
    assert np.array_equal(ids.cpu().numpy(), o_ids)
    assert np.allclose(dist.cpu().numpy(), o_dist, rtol=1e-6)
    assert np.array_equal(st[:, :2].cpu().numpy(), o_st[:, :2])
    return st.cpu().numpy()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("d", [4, 60, 64, 68, 128, 132, 192, 256, 260, 516])
def test_dimensions(d, prec):
    """Half-warp and whole-warp gathers, lanes with and without coordinates; more and
    fewer new nodes than a gather round, through the table and the CSR lists; seeds
    repeated within a batch and across batches of seeds."""
    X = synth.small_integers(700, d, high=200 if d > 64 else 9, seed=d)
    Q = synth.small_integers(9, d, high=200 if d > 64 else 9, seed=d + 1)
    nbr, ln = oracle.knng(X, 45)
    g = oracle.adjust_degree(nbr, ln, 20, 45)
    rng = np.random.default_rng(d)
    seeds = rng.integers(0, 700, size=(9, 40)).astype(np.int32)
    seeds[:, 5] = seeds[:, 3]
    seeds[:, 36] = seeds[:, 2]
    for k, e_s, eps, padded in ((10, 7, 0.1, 7), (10, 20, 0.2, 24), (3, 40, 0.05, 40), (10, 0, 0.1, 0), (40, 0, 0.02, 0)):
        _compare(X, Q, g, seeds, k, e_s, eps, padded, prec)
    _compare(X, Q, g, seeds, 10, 20, 0.2, 20, prec, cap=5)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("d", [384, 388, 448, 512, 576, 1020, 1024])
def test_long_vectors(d, prec):
    """The same where a lane holds up to sixteen quads of a vector, whole and partial."""
    test_dimensions(d, prec)


@pytest.mark.parametrize("n", [2, 513, 6000, 20000])
def test_everything_visited(n):
    """eps = inf visits every node: from a table that stays nearly empty to one that
    overflows into the bitmap, and candidate sets that fill the head, the overflow and the
    pool and are refilled from each."""
    X = synth.small_integers(n, 8, high=64, seed=n)
    Q = synth.small_integers(5, 8, high=64, seed=n + 1)
    nbr, ln = oracle.knng(X, min(16, n - 1))
    g = oracle.adjust_degree(nbr, ln, min(8, n - 1), min(16, n - 1))
    seeds = np.tile(np.arange(min(n, 6), dtype=np.int32), (5, 1))
    _compare(X, Q, g, seeds, min(10, n), 0, np.inf, 0, 0)
    st = _compare(X, Q, g, seeds, min(10, n), 24, np.inf, 24, 0)
    assert (st[:, 3] == 0).all()


@pytest.mark.parametrize("n", [(1 << 23) - 1, 1 << 23, (1 << 23) + 1])
def test_visited_set_at_the_widest_tags_and_beyond(n):
    """The last size whose ids fit a bucket number and 14 tag bits, and the table of ids
    above it: 12,000 linked nodes spread over the ids up to n - 1, rows of more than 32
    entries, repeated seeds, few and all nodes visited (the tables and then the bitmap),
    several queries per warp of a single CTA's workspace."""
    from paper_1810_07355_gb300 import onng
    rng = np.random.default_rng(n % 1000)
    some = np.unique(np.concatenate([rng.integers(0, n, size=12_000), [0, 1, n // 2, n - 2, n - 1]])).astype(np.int32)
    m = len(some)
    deg = np.zeros(n, np.int64)
    deg[some] = np.where(np.arange(m) % 50 == 0, 75, 25)
    ptr = np.concatenate([[0], np.cumsum(deg)])
    col = np.concatenate([some[rng.choice(m, deg[i], replace=False)] for i in some])
    X = np.zeros((n, 4), np.float32)
    X[some] = rng.integers(0, 64, size=(m, 4))
    Q = rng.integers(0, 64, size=(14, 4)).astype(np.float32)
    seeds = some[rng.integers(0, m, size=(14, 9))]
    seeds[:, 4] = seeds[:, 1]
    idx = onng.Index(_dev(ptr), _dev(col), _dev(X))
    cta = 1024 + 4 * ((n + 8191) // 8192 * 1024 + 16384 * 4 + 16384 * 8)

    class OneCta:
        def get(self, need, device):
            return torch.full((cta,), 0xA5, dtype=torch.uint8, device=device)
    for k, e_s, eps, padded in ((10, 0, np.inf, 0), (10, 30, 0.3, 0), (40, 0, 0.1, 0), (10, 20, np.inf, 20), (5, 20, 0.2, 20)):
        if padded:
            idx.with_adjacency(padded)
        for workspace in (None, OneCta()):
            ids, dist, st = onng.search(idx, _dev(Q), k, e_s, eps, _dev(seeds), workspace=workspace)
            o_ids, o_dist, o_st = oracle.search(ptr, col, X, Q, k, e_s, np.float32(eps), seeds)
            assert np.array_equal(ids.cpu().numpy(), o_ids)
            assert np.allclose(dist.cpu().numpy(), o_dist, rtol=1e-6)
            assert np.array_equal(st[:, :2].cpu().numpy(), o_st[:, :2]) and (st[:, 3] == 0).all()


@pytest.mark.parametrize("distinct", [1, 2, 5, 32])
def test_repeated_seeds(distinct):
    """Seeds that repeat few ids over a whole batch and over several: each counts once."""
    X = synth.small_integers(400, 12, high=9, seed=3)
    Q = synth.small_integers(16, 12, high=9, seed=4)
    nbr, ln = oracle.knng(X, 20)
    g = oracle.adjust_degree(nbr, ln, 10, 20)
    rng = np.random.default_rng(distinct)
    some = np.stack([rng.permutation(400)[:distinct] for _ in range(16)])
    seeds = np.take_along_axis(some, rng.integers(0, distinct, size=(16, 64)), 1).astype(np.int32)
    for padded in (0, 20):
        _compare(X, Q, g, seeds, 10, 20, 0.1, padded, 0)


def _algorithm1(g, X, q, k, e_s, eps, seeds):
    """Algorithm 1 a batch at a time (the seeds, then a node's scanned neighbours), with
    IEEE comparisons and a NaN distance ordered after every number (ties by id): ids and
    distances of R, distance computations, expansions."""
    def key(i):
        d2 = float(((X[i] - q) ** 2).sum())
        return (np.inf if np.isnan(d2) else d2, int(i), d2)
    f2 = (1.0 + float(np.float32(eps))) ** 2
    R, S, seen, r2, bound, ndc, nexp = [], [], set(), np.nan, np.inf, 0, 0
    batch, rset = list(dict.fromkeys(seeds.tolist())), False
    while True:
        init = nexp == 0
        new = [key(i) for i in batch if i not in seen]
        seen.update(batch)
        ndc += len(new)
        for c in new:
            if init or not rset or c[2] <= r2:
                R = sorted(R + [c])[:k]
                if not init and len(R) == k:
                    rset, r2 = True, R[-1][2]
        if rset:
            bound = r2 * f2
        S = sorted(S + [c for c in new if c[2] <= bound])
        if not S or S[0][2] > bound:
            return [c[1] for c in R], [np.sqrt(c[2]) for c in R], ndc, nexp
        node, nexp = S.pop(0)[1], nexp + 1
        batch = g[1][g[0][node]:g[0][node + 1]][:e_s].tolist()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("padded", [0, 20])
@pytest.mark.parametrize("nan", ["eps", "rows"])
def test_nan_bound(nan, padded, prec):
    """A NaN eps of some queries, or NaN coordinates that reach the k-th result, make the
    bound NaN in the middle of a search: nothing is pushed from then on, the candidates
    left are expanded, and the other queries are as ever."""
    from paper_1810_07355_gb300 import onng
    rng = np.random.default_rng(5)
    X = synth.small_integers(600, 8, high=9, seed=1)
    Q = synth.small_integers(24, 8, high=9, seed=2)
    nbr, ln = oracle.knng(X, 30)
    g = oracle.adjust_degree(nbr, ln, 12, 30)
    seeds = rng.integers(0, 600, size=(24, 6)).astype(np.int32)
    eps = np.full(24, 0.1, np.float32)
    if nan == "eps":
        eps[::3] = np.nan
    else:
        X[rng.integers(0, 600, size=200), 3] = np.nan
    idx = onng.Index(_dev(g[0].astype(np.int64)), _dev(g[1].astype(np.int32)), _dev(X))
    if padded:
        idx.with_adjacency(padded)
    ids, dist, st = onng.search(idx, _dev(Q), 10, 20, 0.1, _dev(seeds), eps_q=_dev(eps), precision=prec, k_rerank=10)
    ids, dist, st = ids.cpu().numpy(), dist.cpu().numpy(), st.cpu().numpy()
    for r in range(24):
        o_ids, o_dist, ndc, nexp = _algorithm1(g, X, Q[r], 10, 20, eps[r], seeds[r])
        m = len(o_ids)
        assert np.array_equal(ids[r, :m], o_ids) and (ids[r, m:] == -1).all()
        assert np.allclose(dist[r, :m], o_dist, rtol=1e-6, equal_nan=True)
        assert tuple(st[r, :2]) == (ndc, nexp)


@pytest.mark.parametrize("d", [20, 128, 132, 256, 260, 516, 960])
def test_fp8_products_are_rounded(d):
    """A stored vector is the float32 product of scale and code: a query equal to it is at
    distance 0 exactly (the probe's nearest-seed feature is the log of 1e-6)."""
    import ctypes as C

    from paper_1810_07355_gb300 import onng
    rng = np.random.default_rng(d)
    X = (100.0 * rng.random((300, d))).astype(np.float32)
    Q = oracle.fp8_quantize(X)[2][:64]
    idx = onng.Index(_dev(np.zeros(301, np.int64)), _dev(np.zeros(1, np.int32)), _dev(X)).with_fp8()
    Qd, seeds = _dev(Q), _dev(np.stack([np.arange(64), np.arange(64) + 100], 1).astype(np.int32))
    lib, p, ic = onng.load(), onng._Params(2, 0, 0.1, onng.PREC_FP8, 2, 1, 0), idx._c()
    ws = torch.empty(lib.onng_search_workspace_bytes(64, C.byref(ic), C.byref(p)), dtype=torch.uint8, device="cuda")
    feat = torch.empty((64, 16), device="cuda")
    onng._check(lib.onng_search_probe(C.byref(ic), onng._ptr(Qd), 64, C.byref(p), onng._ptr(seeds), 2, 0.9, onng._ptr(feat), None,
                                      onng._ptr(ws), ws.numel(), onng._stream()))
    f = feat.cpu().numpy()
    assert np.abs(f[:, 1] - np.log(1e-6)).max() < 1e-4
    want = np.sqrt(((oracle.fp8_quantize(X)[2][100:164].astype(np.float64) - Q) ** 2).sum(1))
    assert np.allclose(np.exp(f[:, 2]) * 1e-6, want, rtol=1e-4)
