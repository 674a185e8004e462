"""Ranks handed in on both sides of the size where they are written in one pass
or scattered first (launch_import_ranks): they come back as they were, and the
contributions lead to the ranks of one sweep of Eq. 1 on the host, also on a
graph whose internal order is far from the caller's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# one sweep of Eq. 1: the fixed-point sum is off by at most deg * 2^-62 and the
# oracle's FP64 sum by deg * 2^-53 of a sum below 1: under 1e-12 at these degrees
ONE_SWEEP = 1e-12


@pytest.mark.parametrize("n", [3 << 20, (3 << 20) + 1, (1 << 24) + 5])
def test_ranks_in_either_form(n):
    import torch

    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(n)
    # out-degrees without order in the ids, so the internal order is a shuffle
    src = rng.permutation(n).astype(np.int32)[(rng.random(2 * n) ** 3 * n).astype(np.int64)]
    dst = rng.integers(0, n, 2 * n).astype(np.int32)
    r = rng.random(n) ** 4
    r[rng.random(n) < 0.1] = 0.0
    r /= r.sum()
    G = pr.Graph.from_edges(n, src, dst)
    G.set_ranks_device(torch.from_numpy(r).cuda())
    assert np.array_equal(G.ranks(), r)
    G.update("nd", max_iter=1)
    ref, _ = oracle.Graph(n, src, dst).update("nd", r_prev=r, max_iter=1)
    assert np.max(np.abs(G.ranks() - ref)) < ONE_SWEEP
