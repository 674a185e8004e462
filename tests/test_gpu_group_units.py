"""The gather unit that a group picks by the slots of an update's members, and
the host-driven sweeps that are launched ahead of the last one's outcome: the
bits and statistics of a graph updated alone, and of the other loops."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def make(lib, n, m, rng):
    src = (n * rng.random(m) ** 3).astype(np.int32)
    dst = (n * rng.random(m) ** 3).astype(np.int32)
    G = lib.Graph.from_edges(n, src, dst)
    G.update("static")
    r0 = G.ranks()
    k = 500
    G.apply_batch(src[:k], dst[:k], rng.integers(0, n, k), rng.integers(0, n, k))
    return G, r0


def run(update, graphs, r0):
    for G, r in zip(graphs, r0):
        G.set_ranks(r)
    st = update()
    return [G.ranks() for G in graphs], [(s.iterations, s.delta_R, s.vertices_ever_affected, s.vertices_processed,
                                          s.edges_processed) for s in st]


def test_units_by_size_give_the_bits_of_solo_runs():
    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(5)
    pairs = [make(pr, n, m, rng) for n, m in ((700001, 19 << 20), (600011, 19 << 20), (9001, 200000))]
    graphs, r0 = [p[0] for p in pairs], [p[1] for p in pairs]
    grp = pr.Group(graphs)
    host = {m: dict(loop="host", direction=None if m == "nd" else "pull") for m in ("dfp", "df", "nd")}
    assert grp.tuning().steps_per_unit == 4
    try:
        for method in ("dfp", "df", "nd"):
            # all of them, two small enough for the smaller unit, all again
            for sub in ([0, 1, 2], [0, 2], [2, 1, 0]):
                gs, rs = [graphs[i] for i in sub], [r0[i] for i in sub]
                want = run(lambda: [G.update(method, **host[method]) for G in gs], gs, rs)
                got = run(lambda: list(grp.update_members(sub, method).values()), gs, rs)
                assert all(np.array_equal(a, b) for a, b in zip(got[0], want[0])), (method, sub)
                assert got[1] == want[1], (method, sub)
        want = run(lambda: [G.update("dfp", **host["dfp"]) for G in graphs], graphs, r0)
        got = run(lambda: grp.update("dfp", loop="host"), graphs, r0)
        assert all(np.array_equal(a, b) for a, b in zip(got[0], want[0])) and got[1] == want[1]
    finally:
        grp.close()


@pytest.mark.parametrize("method", ["static", "nd", "dt", "df", "dfp"])
def test_host_loop_stops_where_the_others_do(method):
    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(6)
    pair = make(pr, 20011, 300000, rng)
    for kw in (dict(max_iter=1), dict(max_iter=2), dict(max_iter=3), dict(tau=1.0), dict(tau=1e-3), {}):
        out = []
        for opt in (dict(loop="host"), dict(loop="host", time_sweeps=True), dict(loop="device")):
            if method == "dt" and opt.get("loop") == "device":
                opt = dict(time_sweeps=True)
            out.append(run(lambda: [pair[0].update(method, **opt, **kw)], pair[:1], pair[1:]))
        for o in out[1:]:
            assert np.array_equal(o[0][0], out[0][0][0]), (method, kw)
            assert o[1] == out[0][1], (method, kw)
