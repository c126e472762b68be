"""Dynamic Frontier calls whose marking launch leaves its marks to a pull (more than 4 n^2 / m
affected vertices): every row longer than one edge pulls inside that launch, so the list that
the pulls extend is checked for its length, for repeated vertices and against the oracle's
affected set, and the ranks bit for bit against one persistent launch, over many updates."""
import numpy as np
import pytest

import __graft_entry__
import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def prdf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf as mod

    mod.load()
    return mod


@pytest.mark.parametrize("batched", [False, True])
@pytest.mark.parametrize("max_iter", [500, 1])
def test_pulls_of_the_marking_launch(prdf, max_iter, batched):
    g = synth.rmat(14, 16, seed=81)
    p = prdf.pr_params_default()
    p.max_iter = max_iter
    split = []
    for s in (1, 0):
        h = prdf.Graph.batched([g.n, 3], g.src, g.dst, p) if batched else prdf.Graph(g.n, g.src, g.dst, p)
        # bin_lo 1, no groups, 32-edge chunks: every row of two edges or more is in the last tier;
        # dense_div 1: the affected set is never dense, so the marking launch goes on until it defers
        t = h.tuning()
        h.set_tuning(1, t.bin_hi, 1, t.blocks_per_sm, s, 0, 32, 0)
        split.append(h)
    G = oracle.Graph.build(g.n + (3 if batched else 0), g.src, g.dst)
    R, _ = oracle.static_pr(oracle.Graph.build(g.n, g.src, g.dst))
    if batched:
        R = np.concatenate([R, np.full(3, 1 / 3)])
    bs = synth.BatchStream(g, seed=82)
    for _ in range(12):
        b = bs.next(3e-3)
        H, ed, ei = G.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
        got = []
        for h in split:
            h.set_ranks(R)
            h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
            st = h.frontier()
            a = np.sort(h.affected())
            assert a.size == st.affected_final == np.unique(a).size
            got.append((st.iterations, a, h.ranks().copy()))
        assert got[0][0] == got[1][0]
        assert np.array_equal(got[0][1], got[1][1]) and np.array_equal(got[0][2], got[1][2])
        if not batched:
            _, aff, _ = oracle.df_sync(G, H, ed, ei, R, oracle.Params(max_iter=max_iter))
            assert np.array_equal(got[0][1], np.nonzero(aff)[0])
        G, R = H, got[0][2]
    for h in split:
        h.close()
