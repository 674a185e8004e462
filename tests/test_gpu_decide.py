"""Pull sweeps that look up the membership of rows outside the stay set ahead of
the gather (k_decide): the bits and statistics of the device loop, which does
not, on graphs of at least 2^22 vertices with a small batch, hub rows longer
than the warp walks and a ragged last chunk."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra,batch", [(0, 30), (37, 30), (37, 3000)])
def test_rows_decided_ahead_give_the_same_bits(extra, batch):
    import paper_2401_15870_gb300 as pr
    n = (1 << 22) + extra
    src, dst = synth.rmat(22, 16 << 22, 5)
    rng = np.random.default_rng(batch)
    G = pr.Graph.from_edges(n, src, dst)
    G.update("static")
    r0 = G.ranks()
    k = rng.integers(0, src.size, batch // 5)
    G.apply_batch(src[k], dst[k], rng.integers(0, n, batch), rng.integers(0, n, batch))
    for method, kw in (("dfp", {}), ("dfp", dict(tau_p=1e-8)), ("dfp", dict(measure="contrib")), ("df", {})):
        out = []
        for opt in (dict(loop="host"), dict(loop="host", direction="pull"), dict(loop="device")):
            G.set_ranks(r0)
            st = G.update(method, **opt, **kw)
            out.append((G.ranks(), (st.iterations, st.converged, st.delta_R, st.vertices_ever_affected,
                                    st.vertices_processed, st.edges_processed)))
        for o in out[1:]:
            assert np.array_equal(o[0], out[0][0]), (method, kw)
            assert o[1] == out[0][1], (method, kw)
