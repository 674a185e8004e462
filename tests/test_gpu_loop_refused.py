"""One graph's one-kernel loop refused at its launch (pr_debug_fail_loop, no
device is faulted), as it is where a process may not use every SM: the update
runs in the loop that the graph's size takes without it, by default and when the
loop was asked for, with the same bits and statistics; the next one runs in it
again."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

# in-CSR slots: below PR_ONE_KERNEL_SLOTS, and up to three times as many (the
# CUDA graph without it)
SIZES = [(12, 8), (17, 8)]


@pytest.fixture
def lib():
    import paper_2401_15870_gb300 as pr
    yield pr
    pr.pr_debug_fail_loop(0)


@pytest.mark.parametrize("scale,ef", SIZES)
@pytest.mark.parametrize("method", ["static", "nd", "df", "dfp"])
@pytest.mark.parametrize("loop", [None, "one"])
def test_a_refused_loop_falls_back(lib, scale, ef, method, loop):
    n = 1 << scale
    src, dst = synth.rmat(scale, ef * n, 3)
    G = lib.Graph.from_edges(n, src, dst)
    G.update("static")
    r0 = G.ranks()
    cs, cd = synth.unique_edges(src, dst)
    G.apply_batch(*synth.batch(n, cs, cd, 200, 4))

    def run(refused):
        G.set_ranks(r0)
        lib.pr_debug_fail_loop(1 if refused else 0)
        k0 = lib.pr_kernel_launches()
        st = G.update(method, loop=loop)
        launched = lib.pr_kernel_launches() - k0
        return G.ranks(), (st.iterations, st.converged, st.delta_R, st.vertices_ever_affected, st.vertices_processed,
                           st.edges_processed), launched
    first, refused, again = run(False), run(True), run(False)
    for other in (refused, again):
        assert np.array_equal(other[0], first[0]) and other[1] == first[1]
    assert first[2] == again[2] == 1
    # the two-barrier kernel, or the CUDA graph with three kernels an iteration
    graph = loop is None and scale > 12
    assert refused[2] == (2 + 3 * refused[1][0] if graph else 1)


def test_a_group_of_one_falls_back(lib):
    n = 1 << 12
    src, dst = synth.rmat(12, 8 * n, 5)
    G = lib.Graph.from_edges(n, src, dst)
    G.update("static")
    r0 = G.ranks()
    q = lib.Group([G])
    try:
        out = []
        for refused in (0, 1):
            G.set_ranks(r0)
            lib.pr_debug_fail_loop(refused)
            st = q.update("nd")
            out.append((G.ranks(), st[0].iterations))
        assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    finally:
        q.close()
