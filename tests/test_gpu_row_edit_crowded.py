"""Rows that take more insertions than a chunk has slots (edit_crowd): all in
one gap of a row that was emptied, in front of the first or behind the last
element, in a few gaps of many chunks, with deletions beside them; by batches of
the small and the large path, against the edge sets exactly.  And that such
a batch takes about as long as one of the same size spread over the row."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 1 << 20
HUB = 500000       # its id lies in the middle of its neighbours'


def hub_graph(k, seed, into):
    """A hub with k neighbours (out-edges, or in-edges when `into`)."""
    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(seed)
    far = np.sort(rng.choice(np.delete(np.arange(N, dtype=np.int32), HUB), k, replace=False))
    hub = np.full(k, HUB, np.int32)
    src, dst = (far, hub) if into else (hub, far)
    return pr.Graph.from_edges(N, src, dst, keep_order=True), far


def row(G, into):
    r = G.rows(1 if into else 0, np.array([HUB]))[1]
    return r[r != HUB]


def apply(G, into, dels, ins):
    e = [np.full(x.size, HUB, np.int32) for x in (dels, ins)]
    pairs = ((dels, e[0], ins, e[1]) if into else (e[0], dels, e[1], ins))
    G.apply_batch(*[np.ascontiguousarray(x, np.int32) for x in pairs])


def check(G, into, want):
    assert np.array_equal(row(G, into), np.sort(want))
    # the other direction: the hub is in the rows of exactly these vertices
    off, adj = G.rows(0 if into else 1, np.arange(N))
    has = np.add.reduceat(adj == HUB, off[:-1])
    has[HUB] = 0
    assert np.array_equal(np.nonzero(has)[0], np.sort(want))


# left of the row: nothing, its first / last / both ends, a few in the middle,
# most of it but for one wide gap, every 700th
KEEP = {
    "none": lambda a: a[:0], "first": lambda a: a[:1], "last": lambda a: a[-1:], "ends": lambda a: a[[0, -1]],
    "middle": lambda a: a[a.size // 2:a.size // 2 + 40],
    "gap": lambda a: np.r_[a[:a.size // 3], a[a.size // 3 + a.size // 2:]],
    "every 700th": lambda a: a[::700],
}


CASES = [(k, keep, into) for k in (1025, 2500, 16000, 100000) for keep in KEEP for into in (False, True)]
CASES += [(1000000, keep, False) for keep in ("none", "last", "gap")]


@pytest.mark.parametrize("k,keep,into", CASES)
def test_a_row_refilled_through_few_gaps(k, keep, into):
    G, far = hub_graph(k, k, into)
    left = KEEP[keep](far)
    gone = np.setdiff1d(far, left)
    apply(G, into, gone, gone[:0])
    check(G, into, left)
    # refill; every third of the row's rest goes at the same time
    drop = left[1::3]
    apply(G, into, drop, gone)
    check(G, into, np.r_[np.setdiff1d(left, drop), gone])
    # and once more with other ids than before, in the room that is left
    free = np.setdiff1d(np.arange(HUB), far)[: far.size - drop.size]
    now = row(G, into)
    apply(G, into, now[now > far[far.size // 2]], free[:0])
    room = far.size - row(G, into).size
    base = row(G, into)
    apply(G, into, base[::5], free[:room])
    check(G, into, np.r_[np.setdiff1d(base, base[::5]), free[:room]])


def test_one_gap_takes_no_longer_than_many():
    """500,000 insertions into a row of 1,000,000: the same bytes move whether
    they go behind one element or behind every second one."""
    import torch
    G, far = hub_graph(1000000, 9, False)

    def seconds(part):
        s, d = (torch.from_numpy(np.ascontiguousarray(x, np.int32)).cuda() for x in (np.full(part.size, HUB), part))
        e = s[:0]
        took = []
        for _ in range(5):
            G.apply_batch_device(s, d, e, e)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            G.apply_batch_device(e, e, s, d)
            torch.cuda.synchronize()
            took.append(time.perf_counter() - t0)
        return float(np.median(took[1:]))
    spread = seconds(far[::2])
    assert seconds(far[far.size // 2:]) < 4 * spread
    assert seconds(far[:far.size // 2]) < 4 * spread
