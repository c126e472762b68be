"""Single-graph handles in graph-launch mode: every kind of call, in any order, gives what it gives
without (64-bit ranks bit for bit), and a changed tuning or graph is followed."""
import numpy as np
import pytest

import __graft_entry__
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("teleport", [False, True])
@pytest.mark.parametrize("scale", [4, 11, 16])
def test_replayed_calls(scale, teleport):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf

    prdf.load()
    g = synth.rmat(scale, 8, seed=scale)
    bs = synth.BatchStream(g, seed=4)
    p = prdf.pr_params_default()
    p.vertex_order = 2
    if teleport:
        p.dead_end = prdf.PR_DEADEND_TELEPORT
    with prdf.Graph(g.n, g.src, g.dst, p) as a, prdf.Graph(g.n, g.src, g.dst, p) as b:
        b.set_graph_launch(True)
        calls = ("static", "naive", "frontier", "static", "traversal", "naive", "naive", "frontier", "static")
        for k, call in enumerate(calls):
            up = bs.next(1e-2)
            if k == 5:
                for h in (a, b):
                    t = h.tuning()
                    h.set_tuning(4, t.bin_hi, t.dense_div, 1, 1, 0, 128, 16)
            if k == 7:
                for h in (a, b):
                    t = h.tuning()
                    h.set_tuning(4, t.bin_hi, t.dense_div, 1, 0, 0, 128, 16)
            out = []
            for h in (a, b):
                h.apply(up.del_src, up.del_dst, up.ins_src, up.ins_dst)
                st = getattr(h, call)()
                out.append((st.iterations, st.converged, st.affected_final, st.vertices_processed, st.last_delta))
            assert np.array_equal(a.ranks(), b.ranks()), (k, call)
            assert out[0][:3] == out[1][:3] and out[0][4] == out[1][4], (k, call)
            if call in ("static", "naive"):
                assert out[0] == out[1]
