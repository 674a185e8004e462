"""The radix sort's digit widths and tile edges (through graph building, whose
keys are two vertex ids) and the frontier expansion (through the affected sets),
exactly against the oracle: ids of 1 to 21 bits, edge counts around a tile's
8192 keys, hubs over many tiles, levels of one vertex, marked targets."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def same_csr(G, O):
    for mine, ref in ((G.out_csr(), O.out_csr()), (G.in_csr(), O.in_csr())):
        assert np.array_equal(mine[0], ref[0])
        assert np.array_equal(mine[1], ref[1])


# 2 x bits = 2 .. 42: one to five passes; n + m around one and two tiles
@pytest.mark.parametrize("n,m", [(1, 0), (2, 3), (3, 8), (31, 400), (33, 8159), (64, 8128), (700, 8192 - 700),
                                 (1025, 8193 - 1025), (5000, 16384 - 4999), (40000, 70001), (70001, 5),
                                 (1100001, 300000)])
def test_graphs_sorted_over_every_digit_width(n, m):
    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(n + m)
    src, dst = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    same_csr(pr.Graph.from_edges(n, src, dst), oracle.Graph(n, src, dst))


def star(n, rng):   # one vertex to all, and all to another
    a = np.arange(n)
    return np.concatenate([np.zeros(n), a]), np.concatenate([a, np.full(n, n - 1)])


def path(n, rng):
    return np.arange(n - 1), np.arange(1, n)


def dense(n, rng):
    return rng.integers(0, n, 30 * n), rng.integers(0, n, 30 * n)


@pytest.mark.parametrize("n,make", [(40000, star), (700, path), (3000, dense)], ids=["star", "path", "dense"])
def test_affected_sets_match_the_oracle(n, make):
    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(n)
    src, dst = (x.astype(np.int32) for x in make(n, rng))
    G, O = pr.Graph.from_edges(n, src, dst), oracle.Graph(n, src, dst)
    for dels, ins in ((src.size // 2, 1), (3, 2000), (0, 1)):
        at = rng.integers(0, src.size, min(dels, 40))
        b = (src[at], dst[at], rng.integers(0, n, ins).astype(np.int32), rng.integers(0, n, ins).astype(np.int32))
        G.apply_batch(*b)
        O.apply_batch(*b)
        assert np.array_equal(G.initial_affected(), O.initial_affected())
        assert np.array_equal(G.dt_affected(), O.dt_affected())
