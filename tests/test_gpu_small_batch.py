"""Batches of up to 16384 edges (k_small_keys, k_small_ingest, k_small_copy,
k_small_edit) against the oracle's edge sets and effective change, exactly, at
the sizes where the sort changes shape, on rows shorter and longer than a
chunk (1024 elements), rows with few and many changes, rows that overflow."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

N = 5003
# one sweep of Eq. 1 from the same ranks: rounding of the fixed-point and FP64 sums
ONE_SWEEP = 1e-12


def make():
    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(7)
    src = rng.integers(0, N, 12 * N).astype(np.int32)
    dst = rng.integers(0, N, 12 * N).astype(np.int32)
    # two long rows in each direction, one of them just below a chunk
    hub = np.arange(N, dtype=np.int32)
    src = np.concatenate([src, np.full(4000, 11), hub[:1020], np.full(1015, 13)]).astype(np.int32)
    dst = np.concatenate([dst, hub[:4000], np.full(1020, 17), hub[1000:2015]]).astype(np.int32)
    src, dst = np.concatenate([src, hub[:3000]]), np.concatenate([dst, np.full(3000, 19, np.int32)])
    G, O = pr.Graph.from_edges(N, src, dst), oracle.Graph(N, src, dst)
    G.update("static")
    return G, O, src, dst


def check(G, O, r0):
    for mine, ref in ((G.out_csr(), O.out_csr()), (G.in_csr(), O.in_csr())):
        assert np.array_equal(mine[0], ref[0])
        assert np.array_equal(mine[1], ref[1])
    ref, _ = O.update("nd", r_prev=r0, max_iter=1)
    G.update("nd", max_iter=1)
    assert np.max(np.abs(G.ranks() - ref)) < ONE_SWEEP


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("size", [1, 2, 31, 33, 1023, 1024, 1025, 2049, 4096, 4097, 8193, 16383, 16384, 16385])
def test_small_batch_matches_the_oracle(size, device):
    import torch
    G, O, src, dst = make()
    rng = np.random.default_rng(size)
    for step in range(2):
        nd = size // 3
        at = rng.integers(0, src.size, nd)
        ds, dd = src[at].copy(), dst[at].copy()
        is_ = rng.integers(0, N, size - nd).astype(np.int32)
        id_ = rng.integers(0, N, size - nd).astype(np.int32)
        k = (size - nd) // 4
        is_[:k], id_[k:2 * k] = 11, 19              # long rows, many changes each
        is_[2 * k:2 * k + k // 2] = 13              # a row that grows past a chunk
        j = min(nd, k) // 3
        if j:                                       # re-inserted deletions, repeats, a missing edge
            is_[-j:], id_[-j:] = ds[:j], dd[:j]
            ds[j:2 * j], dd[j:2 * j] = ds[:j], dd[:j]
            ds[-1], dd[-1] = 4999, 4998
        if size > 40:
            id_[5] = is_[5]                         # a self-loop
        r0 = G.ranks()
        b = [np.ascontiguousarray(x) for x in (ds, dd, is_, id_)]
        if device:
            G.apply_batch_device(*[torch.from_numpy(x).cuda() for x in b])
        else:
            G.apply_batch(*b)
        O.apply_batch(*b)
        dm, dp = G.effective_delta()
        om, op = O.effective_delta()
        assert np.array_equal(dm, om) and np.array_equal(dp, op)
        check(G, O, r0)
        src, dst = np.concatenate([src, is_]), np.concatenate([dst, id_])


def test_refused_small_batch_keeps_the_last_change():
    import torch

    import paper_2401_15870_gb300 as pr
    G, O, src, dst = make()
    G.apply_batch(src[:3], dst[:3], [1, 2], [2, 4990])
    before = [x.copy() for x in G.effective_delta()]
    e = [np.zeros(9000, np.int32) for _ in range(4)]
    e[3][:] = 1
    e[3][8999] = N
    with pytest.raises(pr.PRError):
        G.apply_batch_device(*[torch.from_numpy(x).cuda() for x in e])
    after = G.effective_delta()
    assert all(np.array_equal(x, y) for x, y in zip(before, after))
    O.apply_batch(src[:3], dst[:3], [1, 2], [2, 4990])
    check(G, O, G.ranks())
