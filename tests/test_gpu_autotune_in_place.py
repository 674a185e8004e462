"""pr_autotune on single sweeps runs each setting as an update would, over the
contributions it gathers where the setting allows (sweep_in_place), and puts
ranks and contributions back: the updates that follow, without ranks handed in
again, give the bits of a twin graph that was not tuned -- also after a batch,
whose sources' contributions it must keep, and on a graph that has no ranks yet."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def run(G, method, **kw):
    st = G.update(method, **kw)
    return G.ranks(), (st.iterations, st.converged, st.delta_R, st.vertices_processed, st.edges_processed)


@pytest.mark.parametrize("scale,ef", [(9, 4), (14, 16)])
@pytest.mark.parametrize("tuned", ["nd", "static"])
@pytest.mark.parametrize("method", ["dfp", "nd", "dt"])
def test_updates_after_tuning_give_the_bits_of_an_untuned_graph(scale, ef, tuned, method):
    import paper_2401_15870_gb300 as pr
    n = 1 << scale
    src, dst = synth.rmat(scale, ef * n, 31)
    cs, cd = synth.unique_edges(src, dst)
    out = []
    for tune in (False, True):
        G = pr.Graph.from_edges(n, src, dst)
        if tune:
            G.autotune("static", reps=1)          # no ranks yet
        G.update("static", loop="host")
        G.apply_batch(*synth.batch(n, cs, cd, n // 20, 32))
        if tune:
            before = G.ranks()
            assert G.autotune(tuned, reps=1).ms_gather > 0
            assert np.array_equal(G.ranks(), before)
        kw = {} if method == "dt" else dict(loop="host")
        out.append([run(G, method, **kw), run(G, "nd", loop="host")])
    for a, b in zip(*out):
        assert np.array_equal(a[0], b[0]) and a[1] == b[1]
