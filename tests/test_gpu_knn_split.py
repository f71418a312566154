"""Exact neighbours where several CTAs share a row block's base tiles, and byte rows of any
dimension on the tensor cores: lists equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1810_07355_gb300 import synth

pytestmark = pytest.mark.gpu


def _knn(X, Q, k, self_offset=-1):
    import torch

    from paper_1810_07355_gb300 import onng
    i, d = onng.knn(torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda(), k, self_offset)
    return i.cpu().numpy(), d.cpu().numpy()


@pytest.mark.parametrize("nq", [1, 16, 17, 33, 65, 127, 129, 300])
@pytest.mark.parametrize("n,d,k", [(131, 8, 5), (6007, 36, 10), (5003, 100, 100), (3001, 128, 40)])
def test_split_sweep_integers(nq, n, d, k):
    """Row blocks of every size, shares of one tile and of many, ragged last tiles;
    tie-heavy integers, so ties by id across the shares' lists."""
    X = synth.small_integers(n, d, high=5, seed=n)
    Q = synth.small_integers(nq, d, high=5, seed=n + 1)
    ids, dist = _knn(X, Q, k)
    o_ids, o_dist = oracle.knn(X, Q, k)
    assert np.array_equal(ids, o_ids)
    assert np.allclose(dist, o_dist, rtol=1e-6, atol=0)


@pytest.mark.parametrize("n,d", [(1500, 32), (4099, 60), (2600, 68), (3333, 124)])
def test_byte_rows_any_dimension(n, d):
    """Self-joins of byte-valued rows on the tensor cores at dimensions that are no
    multiple of 64, with duplicates."""
    X = synth.image_descriptors(n, d=d, clusters=20, seed=n)
    X[n // 2:n // 2 + 50] = X[:50]
    ids, dist = _knn(X, X, 50, 0)
    o_ids, o_dist = oracle.knng(X, 50)
    assert np.array_equal(ids, o_ids)
    assert np.allclose(dist, o_dist, rtol=1e-6, atol=0)


@pytest.mark.parametrize("n,d,k,low", [(4000, 32, 10, 1), (4000, 36, 100, 1), (3000, 64, 40, 2), (5000, 128, 100, 2),
                                       (2600, 68, 5, 0)])
def test_byte_rows_all_tied(n, d, k, low):
    """Rows whose k-th distance is shared by a large part of the base, or by all of it: the
    smallest ids win, in sweeps that start at their own rows and wrap around, and in
    those that several CTAs share."""
    rng = np.random.default_rng(n)
    X = np.full((n, d), 255, np.float32)
    if low:
        X[:, :low] = rng.integers(0, 2, size=(n, low))
    for Q, o in ((X, 0), (X[::9].copy(), -1)):
        ids, dist = _knn(X, Q, k, o)
        o_ids, o_dist = oracle.knn(X, Q, k, np.arange(n) if o == 0 else None)
        assert np.array_equal(ids, o_ids)
        assert np.allclose(dist, o_dist, rtol=1e-6, atol=0)


@pytest.mark.parametrize("nq,n,d", [(40, 5000, 100), (200, 5000, 100), (150, 3000, 260)])
def test_split_sweep_floats(nq, n, d):
    """Float data: every position's length is the float64 one's to float32 rounding of
    the direct difference (at most d + 2 roundings)."""
    rng = np.random.default_rng(d + nq)
    X = rng.normal(size=(n, d)).astype(np.float32)
    Q = rng.normal(size=(nq, d)).astype(np.float32)
    ids, dist = _knn(X, Q, 20)
    _, o_dist = oracle.knn(X, Q, 20)
    assert np.allclose(dist, o_dist, rtol=1e-5, atol=0)
    exact = np.sqrt(((X[ids].astype(np.float64) - Q[:, None].astype(np.float64)) ** 2).sum(2))
    assert np.allclose(dist, exact, rtol=1e-5, atol=0)


@pytest.mark.parametrize("kind,n,d,nq,k", [("int", 6007, 36, 50, 10), ("int", 6007, 256, 300, 100), ("byte", 20_000, 100, 300, 100),
                                           ("byte", 20_000, 128, 257, 10), ("float", 9000, 100, 300, 40),
                                           ("float", 9000, 260, 257, 10), ("int", 3000, 16, 700, 200)])
def test_workspace_sizes(kind, n, d, nq, k):
    """Any workspace from one list per query and share up to the request (and beyond)
    gives the same lists and is not overrun; a smaller one is refused."""
    import torch

    from paper_1810_07355_gb300 import onng
    rng = np.random.default_rng(n + d)
    if kind == "float":
        X = rng.normal(size=(n + nq, d)).astype(np.float32)
    else:
        X = rng.integers(0, 256 if kind == "byte" else 300, size=(n + nq, d)).astype(np.float32)
    X, Q = X[:n], X[n:]
    o_ids, o_dist = oracle.knn(X, Q, k)
    lib = onng.load()
    kc, share, dp, tiles = next(c for c in (32, 64, 128, 256) if k + 16 <= c), 2 if d > 128 else 1, (d + 63) // 64 * 64, -(-n // 128)
    least = 0
    for b in (4 * n, 4 * nq, nq * share * kc * 8, nq * share * 256 * 8, 256, n * dp * 4, nq * dp * 4, tiles * 512, 8 * d, 4 * d,
              tiles * 16):
        least = -(-least // 256) * 256 + b
    ask = lib.onng_knn_workspace_bytes(n, d, nq, k)
    assert least <= ask
    dX, dQ = torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda()
    for size in (least, (2 * least + ask) // 3, ask - 1, ask, 2 * ask, least - 1):
        ws = torch.full((size + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
        ids = torch.empty((nq, k), dtype=torch.int32, device="cuda")
        dist = torch.empty((nq, k), device="cuda")
        st = lib.onng_knn(onng._ptr(dX), n, d, onng._ptr(dQ), nq, k, -1, onng._ptr(ids), onng._ptr(dist), onng._ptr(ws), size,
                          onng._stream())
        assert st == (onng.ONNG_E_WORKSPACE if size < least else onng.ONNG_OK)
        assert (ws[size:] == 0xA5).all()
        if st == onng.ONNG_OK:
            if kind != "float":
                assert np.array_equal(ids.cpu().numpy(), o_ids)
            assert np.allclose(dist.cpu().numpy(), o_dist, rtol=1e-5, atol=0)
