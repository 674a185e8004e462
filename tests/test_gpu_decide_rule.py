"""That k_decide has work in the inputs of test_gpu_decide.py: its rule
(DECIDE_OUT, DECIDE_DEG, DECIDE_N), worked out on the host from the ranks before
and after a sweep, asks for it in a sweep that the update runs, while rows it
decides at once, rows the warp walks and rows it leaves open lie outside the
stay set; and the update that has such a sweep gives the bits of the device
loop, which does not look ahead."""
import os
import re

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TAU_F = TAU_P = 1e-6


def constant(name):
    text = open(os.path.join(ROOT, "paper_2401_15870_gb300", "csrc", "sweep.cu")).read()
    v = re.search(r"constexpr \w+ %s = ([^;]+);" % name, text).group(1)
    a, _, b = v.partition("<<")
    return int(a) << int(b) if b else float(v)


@pytest.mark.parametrize("extra,batch", [(0, 30), (37, 30), (37, 3000)])
def test_the_rule_asks_for_rows_decided_ahead(extra, batch):
    import paper_2401_15870_gb300 as pr
    n = (1 << 22) + extra
    assert n >= constant("DECIDE_N")
    src, dst = synth.rmat(22, 16 << 22, 5)
    rng = np.random.default_rng(batch)
    G = pr.Graph.from_edges(n, src, dst)
    G.update("static")
    r0 = G.ranks()
    k = rng.integers(0, src.size, batch // 5)
    G.apply_batch(src[k], dst[k], rng.integers(0, n, batch), rng.integers(0, n, batch))
    deg = np.diff(G.rows(1, np.arange(n, dtype=np.int32), degrees_only=True))
    m = G.m
    walked = 4 * (4 + 32 * constant("DECIDE_STEPS"))     # slots looked at before a row is left open

    def ranks_after(it):
        G.set_ranks(r0)
        st = G.update("dfp", loop="host", direction="pull", max_iter=it)
        return G.ranks(), st.iterations

    full = ranks_after(500)
    asked = []
    prev = r0
    for it in range(1, min(8, full[1])):                # the sweep after `it` is run too
        cur, _ = ranks_after(it)
        stay = np.abs(cur - prev) > TAU_P * np.maximum(cur, prev)
        prev = cur
        s_edges, s = int(deg[stay].sum()), int(stay.sum())
        if (m - s_edges) > constant("DECIDE_OUT") * m and s_edges * float(n) > constant("DECIDE_DEG") * m * s:
            out = deg[~stay]
            asked.append((it, s / n, int((out <= 16).sum()), int(((out > 16) & (out <= walked)).sum()),
                          int((out > walked).sum())))
    assert asked
    assert all(any(a[k] for a in asked) for k in (2, 3, 4))
    G.set_ranks(r0)
    st = G.update("dfp", loop="device")
    assert np.array_equal(G.ranks(), full[0]) and st.iterations == full[1]
