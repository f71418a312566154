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
