"""A rank call that ends early leaves a usable handle.

The calls are ended by a short limit on the barrier waits, at whatever point the wait that runs out
is; the call returns PR_ERR_DEVICE_TIMEOUT and the next one, without new ranks, must give the
ranks of the graph as it is, whatever the unfinished call had marked, iterated or restarted."""
import numpy as np
import pytest

import __graft_entry__
import oracle
import synth

pytestmark = pytest.mark.gpu

# waits of different lengths run out: the first one of a call, and ones inside its iterations
LIMITS_US = [1, 2, 3, 4, 5, 6, 8, 10, 12, 15, 20, 30]


@pytest.fixture(scope="module")
def prdf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf as mod

    mod.load()
    return mod


def _limit(h, t, us, split):
    h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, split, us)


@pytest.mark.parametrize("first", ["frontier", "traversal", "naive", "static"])
@pytest.mark.parametrize("kind", ["single", "batched", "teleport", "one launch"])
def test_the_next_call_gives_the_graphs_ranks(prdf, kind, first):
    g = synth.rmat(13, 8, seed=91)
    p = prdf.pr_params_default()
    op = oracle.Params()
    if kind == "teleport":
        p.dead_end = prdf.PR_DEADEND_TELEPORT
        op = oracle.Params(dead_end=oracle.TELEPORT)
    split = 0 if kind == "one launch" else 1
    G = oracle.Graph.build(g.n, g.src, g.dst, self_loops=kind != "teleport")
    bs = synth.BatchStream(g, seed=92)
    h = prdf.Graph.batched([g.n, 2], g.src, g.dst, p) if kind == "batched" else prdf.Graph(g.n, g.src, g.dst, p)
    ended = 0
    with h:
        t = h.tuning()
        h.static()
        for k, us in enumerate(LIMITS_US):
            b = bs.next(1e-2)
            h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
            G = G.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)[0]
            _limit(h, t, us, split)
            try:
                getattr(h, first)()
            except prdf.PrdfError as e:
                assert e.status == prdf.PR_ERR_DEVICE_TIMEOUT
                ended += 1
            if k % 2:  # another update between the two
                b = bs.next(1e-2)
                h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
                G = G.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)[0]
            _limit(h, t, 0, split)
            for call in ("frontier", "frontier"):
                assert getattr(h, call)().converged
                # a change of 1e-10 stops both: 2 tau / (1 - alpha) apart at most
                assert np.abs(h.ranks()[:g.n] - oracle.static_pr(G, op)[0]).max() <= 2e-9, (us, call)
    # (one launch an iteration has no barrier to wait at)
    assert ended > 0 or (kind == "one launch" and first in ("naive", "static"))


def test_new_ranks_keep_the_pending_marks(prdf):
    g = synth.rmat(13, 8, seed=93)
    G = oracle.Graph.build(g.n, g.src, g.dst)
    R, _ = oracle.static_pr(G)
    b = synth.BatchStream(g, seed=94).next(1e-3)
    H, ed, ei = G.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
    with prdf.Graph(g.n, g.src, g.dst) as h:
        t = h.tuning()
        h.set_ranks(R)
        h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
        _limit(h, t, 1, 1)
        with pytest.raises(prdf.PrdfError):
            for _ in range(20):
                h.frontier()
                h.set_ranks(R)
                h.apply(b.ins_src, b.ins_dst, b.del_src, b.del_dst)
                h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
        _limit(h, t, 0, 1)
        h.set_ranks(R)
        st = h.frontier()
        R_df, aff, st_df = oracle.df_sync(G, H, ed, ei, R)
        assert np.abs(h.ranks() - R_df).max() <= 1e-9
        assert set(np.nonzero(aff)[0].tolist()) <= set(h.affected().tolist()) and st.affected_final < g.n
