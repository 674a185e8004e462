"""Ranks handed in on the device (k_check_ranks, k_import_ranks): what comes
back, the contributions they lead to, and what is refused."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

# one sweep of Eq. 1: the fixed-point sum is off by at most deg * 2^-62 and the
# oracle's FP64 sum by deg * 2^-53 of a sum below 1: under 1e-12 at these degrees
ONE_SWEEP = 1e-12


@pytest.mark.parametrize("n", [1, 2, 31, 33, 255, 257, 4097, 700001])
def test_imported_ranks_and_their_contributions(n):
    import torch

    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(n)
    src, dst = (rng.integers(0, n, 4 * n).astype(np.int32) for _ in range(2))
    r = rng.random(n) ** 4
    r[rng.random(n) < 0.1] = 0.0
    r /= max(r.sum(), 1e-300)
    G = pr.Graph.from_edges(n, src, dst)
    G.set_ranks_device(torch.from_numpy(r).cuda())
    assert np.array_equal(G.ranks(), r)
    G.update("nd", max_iter=1)
    ref, _ = oracle.Graph(n, src, dst).update("nd", r_prev=r, max_iter=1)
    assert np.max(np.abs(G.ranks() - ref)) < ONE_SWEEP


@pytest.mark.parametrize("n", [1, 255, 300001])
def test_bad_ranks_are_refused_and_change_nothing(n):
    import torch

    import paper_2401_15870_gb300 as pr
    G = pr.Graph.from_edges(n, np.zeros(0, np.int32), np.zeros(0, np.int32))
    good = np.full(n, 1.0 / n)
    G.set_ranks_device(torch.from_numpy(good).cuda())
    for at in (0, n // 2, n - 1):
        for bad in (-1e-300, -np.inf, np.inf, np.nan, 2.5):
            r = good.copy()
            r[at] = bad
            with pytest.raises(pr.PRError):
                G.set_ranks_device(torch.from_numpy(r).cuda())
            assert np.array_equal(G.ranks(), good)
