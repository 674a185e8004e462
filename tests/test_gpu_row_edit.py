"""Rows rewritten in place (k_edit_short, k_edit_long) by batches of more than
16384 edges, against the oracle's edge sets exactly: rows at the borders of
64 and 1024 slots, of several chunks, with few and with many changes per chunk,
changes before the first and after the last element and many between two
neighbours, rows that grow or shrink over a border, and repeated batches that
use the slack up."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

N = 30011
# one sweep of Eq. 1 from the same ranks: rounding of the fixed-point and FP64 sums
ONE_SWEEP = 1e-12
DEGREES = [1, 3, 4, 59, 60, 61, 63, 64, 65, 127, 1019, 1020, 1023, 1024, 1025, 2047, 2048, 2049, 5000, 20000]


@pytest.fixture(scope="module")
def start():
    """Out-rows and in-rows of the listed degrees among a sparse random graph."""
    rng = np.random.default_rng(3)
    src = [rng.integers(200, N, 6 * N)]
    dst = [rng.integers(200, N, 6 * N)]
    for k, d in enumerate(DEGREES):
        other = np.sort(rng.choice(np.arange(300, N), d - 1, replace=False))   # the self-loop makes d
        src += [np.full(d - 1, k), other]
        dst += [other, np.full(d - 1, 100 + k)]
    return np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)


def changes(rng, src, dst, per_row, share):
    """Deletions of a share of the listed rows' edges and insertions into them."""
    dels, ins = [], []
    for k in range(len(DEGREES)):
        for col, key in ((src, k), (dst, 100 + k)):
            at = np.nonzero(col == key)[0]
            if at.size:
                dels.append(rng.choice(at, max(1, int(at.size * share)), replace=False))
            y = np.concatenate([rng.integers(200, N, per_row), [0, 1, 150, 199, N - 1, N - 2]])
            y = np.concatenate([y, 15000 + np.arange(per_row // 2)])           # many between two neighbours
            ins.append(np.stack([np.full(y.size, key), y]) if key == k else np.stack([y, np.full(y.size, key)]))
    return np.concatenate(dels), np.concatenate(ins, axis=1).astype(np.int32)


@pytest.mark.parametrize("per_row,share", [(1, 0.0), (4, 0.01), (40, 0.05), (600, 0.3), (2, 0.9)])
def test_rows_edited_in_place_match_the_oracle(start, per_row, share):
    import paper_2401_15870_gb300 as pr
    src, dst = start
    G, O = pr.Graph.from_edges(N, src, dst, keep_order=True), oracle.Graph(N, src, dst)
    G.update("static")
    rng = np.random.default_rng(per_row)
    for step in range(3):
        at, ins = changes(rng, src, dst, per_row, share)
        ds, dd = src[at], dst[at]
        pad = rng.integers(200, N, (2, 20000)).astype(np.int32)                # past the small-batch path
        is_, id_ = np.concatenate([ins[0], pad[0]]), np.concatenate([ins[1], pad[1]])
        r0 = G.ranks()
        G.apply_batch(ds, dd, is_, id_)
        O.apply_batch(ds, dd, is_, id_)
        for mine, ref in ((G.out_csr(), O.out_csr()), (G.in_csr(), O.in_csr())):
            assert np.array_equal(mine[0], ref[0])
            assert np.array_equal(mine[1], ref[1])
        dm, dp = G.effective_delta()
        om, op = O.effective_delta()
        assert np.array_equal(dm, om) and np.array_equal(dp, op)
        ref, _ = O.update("nd", r_prev=r0, max_iter=1)
        G.update("nd", max_iter=1)
        assert np.max(np.abs(G.ranks() - ref)) < ONE_SWEEP
        keep = np.ones(src.size, bool)
        keep[at] = False
        src, dst = np.concatenate([src[keep], is_]), np.concatenate([dst[keep], id_])
