"""Pivot seeds where the pivots are split over a cluster and over tiles: ids equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1810_07355_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,P,n_seed,d", [(1, 127, 10, 32), (1, 1024, 10, 128), (33, 1025, 32, 36), (31, 513, 33, 20),
                                           (17, 4097, 64, 100), (700, 257, 1, 12)])
def test_pivot_split_equals_oracle(nq, P, n_seed, d):
    """Ragged query blocks, tiles and cluster shares; small integers give many ties
    within and across shares (ties by pivot index), one list of each length class."""
    import torch

    from paper_1810_07355_gb300 import onng
    X = synth.small_integers(5000, d, high=4, seed=d)
    Q = synth.small_integers(nq, d, high=4, seed=d + 1)
    s = onng.seeds_pivot(torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda(), P, n_seed)
    assert np.array_equal(s.cpu().numpy(), oracle.seeds_pivot(X, Q, P, n_seed))


@pytest.mark.parametrize("n_seed", [10, 64])
@pytest.mark.parametrize("P", [1024, 4096])
@pytest.mark.parametrize("d", [4, 8, 12, 16, 20])
def test_tiles_of_one_chunk(d, P, n_seed):
    """Rows of at most 16 coordinates, several tiles per CTA (without and with a split over
    a cluster): the pivots come nearer from first to last, so the queries at 0 take new
    nearest ones in every tile while those at P keep the first tile's; the two kinds
    alternate over the warps.  All distances that can be returned are exact."""
    import torch

    from paper_1810_07355_gb300 import onng
    X = synth.small_integers(P, d, high=3, seed=d)
    X[:, 0] = P - np.arange(P)
    for nq in (64, 5000):
        Q = synth.small_integers(nq, d, high=3, seed=d + 1)
        Q[:, 0] = np.where(np.arange(nq) % 2 == 0, 0, P)
        dX, dQ, want = torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda(), oracle.seeds_pivot(X, Q, P, n_seed)
        for _ in range(5):
            assert np.array_equal(onng.seeds_pivot(dX, dQ, P, n_seed).cpu().numpy(), want)


@pytest.mark.parametrize("d", [4, 64, 68, 200])
@pytest.mark.parametrize("P,n_seed", [(1, 1), (1, 64), (31, 40), (63, 10), (64, 64), (65, 10), (127, 33), (128, 64), (129, 64)])
def test_few_pivots(P, n_seed, d):
    """One and two tiles of the few-pivot kernel and the sizes beside them, with ties, more
    seeds than pivots, and rows that are not finite; the sets of queries on both sides of
    each rule."""
    import torch

    from paper_1810_07355_gb300 import onng
    X = synth.small_integers(900, d, high=4, seed=d)
    Q = synth.small_integers(2600, d, high=4, seed=d + 1)
    for nq in (1, 15, 17, 300, 2600):
        s = onng.seeds_pivot(torch.from_numpy(X).cuda(), torch.from_numpy(Q[:nq]).cuda(), P, n_seed)
        assert np.array_equal(s.cpu().numpy(), oracle.seeds_pivot(X, Q[:nq], P, n_seed))
    nan = [int(t) * 900 // P for t in range(0, P, 3)]
    X[nan, d - 1] = np.nan  # such pivots are never taken
    s = onng.seeds_pivot(torch.from_numpy(X).cuda(), torch.from_numpy(Q[:40]).cuda(), P, n_seed).cpu().numpy()
    ids = np.array([t * 900 // P for t in range(P) if t % 3])
    for r in range(40):
        d2 = ((X[ids] - Q[r]) ** 2).sum(1) if len(ids) else np.empty(0)
        want = ids[np.argsort(d2, kind="stable")][:n_seed] if len(ids) else ids
        assert np.array_equal(s[r, :len(want)], want) and (s[r, len(want):] == -1).all()
