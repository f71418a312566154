"""Path and degree adjustment at the row sizes where another kernel or another sorting
network takes over: results and witnesses equal the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _graph(n, hub, seed):
    """A CSR of n rows of 1 .. 40 edges, some of them of `hub` edges; rows by (length, id),
    lengths with many ties."""
    rng = np.random.default_rng(seed)
    deg = rng.integers(1, 41, size=n)
    deg[rng.choice(n, 3, replace=False)] = hub
    rp = np.concatenate([[0], np.cumsum(deg)]).astype(np.int64)
    col, ln = np.empty(rp[-1], np.int32), np.empty(rp[-1], np.float32)
    for i in range(n):
        ids = rng.choice(n - 1, deg[i], replace=False)
        ids = np.where(ids >= i, ids + 1, ids)
        length = rng.integers(1, 60, size=deg[i]).astype(np.float32)
        o = np.lexsort((ids, length))
        col[rp[i]:rp[i + 1]], ln[rp[i]:rp[i + 1]] = ids[o], length[o]
    return rp, col, ln


@pytest.mark.parametrize("n,hub", [(300, 31), (600, 256), (600, 257), (1100, 1024), (1100, 1025), (2500, 2047),
                                   (8400, 8192), (8400, 8193)])
def test_path_rows(n, hub):
    import torch

    from paper_1810_07355_gb300 import onng
    rp, col, ln = _graph(n, hub, hub)
    got = onng.adjust_path(*(torch.from_numpy(v).cuda() for v in (rp, col, ln)), witnesses=True)
    want = oracle.adjust_path(rp, col, ln, witnesses=True)
    for g, w in zip(got, want):
        assert np.array_equal(g.cpu().numpy(), w.astype(g.cpu().numpy().dtype))


@pytest.mark.parametrize("n,k,e_o,e_i", [(700, 31, 31, 31), (700, 64, 33, 1), (1500, 100, 0, 100), (40, 39, 39, 39),
                                         (900, 6, 5, 6)])
def test_degree_rows(n, k, e_o, e_i):
    """kNN widths that are and are not a multiple of four, one to several 32-entry chunks,
    rows of every sorting network, reversed edges onto a hub of more than 512."""
    import torch

    from paper_1810_07355_gb300 import onng
    rng = np.random.default_rng(k)
    nbr = np.empty((n, k), np.int32)
    for i in range(n):
        ids = rng.choice(n - 1, k, replace=False)
        ids = np.where(ids >= i, ids + 1, ids)
        if i > 0 and 0 not in ids:
            ids[rng.integers(0, k)] = 0  # node 0 is a hub
        nbr[i] = ids
    ln = np.sort(rng.integers(1, 40, size=(n, k)).astype(np.float32), axis=1)
    for i in range(n):
        nbr[i] = nbr[i][np.lexsort((nbr[i], ln[i]))]
    got = onng.adjust_degree(torch.from_numpy(nbr).cuda(), torch.from_numpy(ln).cuda(), e_o, e_i)
    want = oracle.adjust_degree(nbr, ln, e_o, e_i)
    for g, w in zip(got, want[:3]):
        assert np.array_equal(g.cpu().numpy(), w.astype(g.cpu().numpy().dtype))


def test_row_order_of_nodes_without_in_edges():
    """Only the rows of neighbours are searched by length: a node that nothing points to
    may hold its edges (up to 256) in any order, or lengths that are no numbers behind
    them, and loses the edges the rule says."""
    import torch

    from paper_1810_07355_gb300 import onng
    rng = np.random.default_rng(8)
    n, extra = 900, 60
    X = rng.normal(size=(n + extra, 6)).astype(np.float32)
    nbr, ln = oracle.knng(X[:n], 24)
    ptr, col, length = oracle.adjust_degree(nbr, ln, 12, 24)
    ptr, cols, lens = ptr.tolist(), [col], [length.astype(np.float32)]
    for i in range(extra):
        deg = [1, 2, 3, 31, 32, 33, 64, 100, 255, 256][i % 10]
        d = np.sqrt(((X[:n] - X[n + i]) ** 2).sum(1))
        c = np.argsort(d, kind="stable")[:deg]
        l = d[c].astype(np.float32)
        if i < 40:
            o = rng.permutation(deg) if i < 30 else np.arange(deg)[::-1]
            c, l = c[o], l[o]
        else:
            l[-max(1, deg // 8):] = np.nan
        ptr.append(ptr[-1] + deg)
        cols.append(c.astype(np.int32))
        lens.append(l)
    ptr, col, length = np.array(ptr, np.int64), np.concatenate(cols), np.concatenate(lens)
    want = oracle.adjust_path(ptr, col, length, witnesses=True)
    got = [t.cpu().numpy() for t in onng.adjust_path(*(torch.from_numpy(a).cuda() for a in (ptr, col, length)), witnesses=True)]
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert np.array_equal(got[2], want[2].astype(np.float32), equal_nan=True)
    assert np.array_equal(got[3], want[3])


@pytest.mark.parametrize("n,deg", [(1, 0), (40, 1), (50, 5), (51, 5), (300, 257), (1100, 1025)])
def test_few_edges_and_workspace_bounds(n, deg):
    """Graphs too small to hold a row of the next size, and those just large enough; the
    call stays within a workspace of exactly the requested size."""
    import ctypes as C

    import torch

    from paper_1810_07355_gb300 import onng
    rng = np.random.default_rng(n)
    rp = np.minimum(np.arange(n + 1) * deg, deg * (n if n < 100 else 5)).astype(np.int64)
    nnz = int(rp[-1])
    col, ln = np.empty(nnz, np.int32), np.empty(nnz, np.float32)
    for i in range(n):
        m = int(rp[i + 1] - rp[i])
        ids = rng.choice(n - 1, m, replace=False) if m else np.empty(0, np.int64)
        ids = np.where(ids >= i, ids + 1, ids)
        length = rng.integers(1, 20, size=m).astype(np.float32)
        o = np.lexsort((ids, length))
        col[rp[i]:rp[i + 1]], ln[rp[i]:rp[i + 1]] = ids[o], length[o]
    want = oracle.adjust_path(rp, col, ln, witnesses=True)
    lib = onng.load()
    size = lib.onng_adjust_path_workspace_bytes(n, nnz)
    ws = torch.full((size + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    d_rp, d_col, d_ln = (torch.from_numpy(v).cuda() for v in (rp, np.append(col, 0).astype(np.int32), np.append(ln, 0).astype(np.float32)))
    o_rp = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    o_col, o_wit = (torch.full((nnz + 1,), -7, dtype=torch.int32, device="cuda") for _ in range(2))
    o_ln = torch.empty(nnz + 1, device="cuda")
    kept = C.c_int64(0)
    onng._check(lib.onng_adjust_path(onng._ptr(d_rp), onng._ptr(d_col), onng._ptr(d_ln), n, onng._ptr(o_rp), onng._ptr(o_col),
                                     onng._ptr(o_ln), C.byref(kept), onng._ptr(o_wit), onng._ptr(ws), size, onng._stream()))
    assert (ws[size:] == 0xA5).all()
    m = kept.value
    assert np.array_equal(o_rp.cpu().numpy(), want[0]) and m == len(want[1])
    assert np.array_equal(o_col[:m].cpu().numpy(), want[1]) and np.array_equal(o_ln[:m].cpu().numpy(), want[2].astype(np.float32))
    assert np.array_equal(o_wit[:nnz].cpu().numpy(), want[3])
