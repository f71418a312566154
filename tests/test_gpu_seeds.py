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
