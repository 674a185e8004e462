"""The one-kernel loop of a single graph whose grid barrier never completes
(pr_debug_fail_loop: a count whose arrivals never come, and a short wait): the
kernel ends by itself and the call returns PR_ETIMEOUT, the graph has no ranks
and a dynamic update is refused; with ranks handed in again the next update gives
the bits of before.  For frontier and every-vertex methods, rows kept in
registers or not, a group of one, and twice in a row."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

ENORANKS, ETIMEOUT = 4, 6


@pytest.fixture
def lib():
    import paper_2401_15870_gb300 as pr
    yield pr
    pr.pr_debug_fail_loop(0)


def graph(lib, n, m, seed):
    rng = np.random.default_rng(seed)
    src, dst = (rng.integers(0, n, m).astype(np.int32) for _ in range(2))
    G = lib.Graph.from_edges(n, src, dst)
    G.update("static")
    r0 = G.ranks()
    G.apply_batch(src[:50], dst[:50], *(rng.integers(0, n, 50).astype(np.int32) for _ in range(2)))
    return G, r0


def result(G, r0, method, loop=None):
    G.set_ranks(r0)
    st = G.update(method, loop=loop)
    return G.ranks(), (st.iterations, st.converged, st.delta_R, st.vertices_ever_affected, st.vertices_processed,
                       st.edges_processed)


# at most one row per thread of 152 blocks of 1024, and more
@pytest.mark.parametrize("n,m", [(1000, 8000), (200003, 100000)])
@pytest.mark.parametrize("method", ["static", "nd", "df", "dfp"])
def test_a_barrier_that_never_completes_is_given_up(lib, n, m, method):
    G, r0 = graph(lib, n, m, 7)
    want = result(G, r0, method)
    for _ in range(2):
        G.set_ranks(r0)
        lib.pr_debug_fail_loop(2)
        with pytest.raises(lib.PRError) as e:
            G.update(method)
        assert e.value.status == ETIMEOUT
        with pytest.raises(lib.PRError) as e:
            G.update("dfp")
        assert e.value.status == ENORANKS
        with pytest.raises(lib.PRError):
            G.ranks()
    for loop in (None, "one", "device"):
        got = result(G, r0, method, loop)
        assert np.array_equal(got[0], want[0]) and got[1] == want[1], loop
    G.update("static")   # and from no ranks at all
    assert np.array_equal(result(G, r0, method)[0], want[0])


def test_a_group_of_one_gives_up_and_recovers(lib):
    G, r0 = graph(lib, 3000, 30000, 8)
    want = result(G, r0, "dfp")
    q = lib.Group([G])
    try:
        for fail in (0, 2, 0):
            G.set_ranks(r0)
            lib.pr_debug_fail_loop(fail)
            if fail:
                with pytest.raises(lib.PRError) as e:
                    q.update("dfp")
                assert e.value.status == ETIMEOUT
            else:
                assert q.update("dfp")[0].iterations == want[1][0]
                assert np.array_equal(G.ranks(), want[0])
    finally:
        q.close()
