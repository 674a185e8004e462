"""The loop with one grid barrier per iteration (loop.cu): the bits and
statistics of the host loop where its work is shared out unevenly -- fewer
rows than blocks, more rows than threads in a block, rows over many 32-quad
words, columns kept in shared memory or not, graphs it hands back."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def star(n, rng):
    return np.arange(n, dtype=np.int32), np.zeros(n, np.int32)


def uniform(per):
    def make(n, rng):
        m = int(n * per)
        return rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
    return make


def skewed(per):
    def make(n, rng):
        m = int(n * per)
        return ((n * rng.random(m) ** 4).astype(np.int32), (n * rng.random(m) ** 4).astype(np.int32))
    return make


# (name, n, edges): one vertex; two rows for 152 blocks; a row that continues
# over 70 words; the same beyond the longest row the loop takes; one row per
# thread just kept and just exceeded (152 x 1024 rows of two quads); columns
# staged and not; hub rows beside many short ones
CASES = [
    ("one", 1, uniform(0)), ("two", 2, uniform(2)), ("star", 9001, star), ("long star", 40001, star),
    ("sparse", 140001, uniform(0.3)), ("sparse more", 330001, uniform(0.1)), ("dense", 3001, uniform(64)),
    ("skewed", 20011, skewed(20)), ("skewed large", 90001, skewed(24)),
]


@pytest.mark.parametrize("name,n,make", CASES, ids=[c[0] for c in CASES])
def test_one_barrier_loop_gives_the_bits_of_the_host_loop(name, n, make):
    import paper_2401_15870_gb300 as pr
    rng = np.random.default_rng(n)
    G = pr.Graph.from_edges(n, *make(n, rng))
    G.update("static", loop="host")
    r0 = G.ranks()
    k = min(500, n)
    rows = G.rows(0, np.arange(min(n, 50)))
    dels = (np.repeat(np.arange(min(n, 50)), np.diff(rows[0])).astype(np.int32)[::3], rows[1][::3])
    G.apply_batch(*dels, rng.integers(0, n, k), rng.integers(0, n, k))
    for method, kw in (("static", {}), ("nd", {}), ("df", {}), ("dfp", {}), ("dfp", dict(tau_p=1e-8)),
                       ("df", dict(measure="contrib")), ("dfp", dict(measure="absolute", tau_f=1e-12, tau_p=1e-12))):
        out = []
        for loop in ("one", "host"):
            G.set_ranks(r0)
            st = G.update(method, loop=loop, **kw)
            out.append((G.ranks(), (st.iterations, st.converged, st.delta_R, st.vertices_ever_affected,
                                    st.vertices_processed, st.edges_processed)))
        assert np.array_equal(out[0][0], out[1][0]), (method, kw)
        assert out[0][1] == out[1][1], (method, kw)
