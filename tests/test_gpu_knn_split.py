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
