"""Graphs in a server: the dense iterations' runs are bounded, and the launch sizes a graph had before
come back with the end of the server."""
import numpy as np
import pytest

import __graft_entry__
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf

    prdf.load()
    return prdf, torch


@pytest.mark.parametrize("slots", [1, 2, 3, 64])
def test_handles_get_their_launch_sizes_back(env, slots):
    prdf, torch = env
    gs = [synth.rmat(12, 8, seed=5 + k) for k in range(2)]
    hs = [prdf.Graph(g.n, g.src, g.dst, None, torch.cuda.Stream().cuda_stream) for g in gs]
    t = hs[1].tuning()
    hs[1].set_tuning(t.bin_lo, t.bin_hi, t.dense_div, 1)
    before = [h.tuning().blocks_per_sm for h in hs]
    for _ in range(2):  # and once more, in another server
        with prdf.Server(slots=slots) as srv:
            for h in hs:
                srv.add(h)
        assert [h.tuning().blocks_per_sm for h in hs] == before
    # a graph that goes first (its server must not touch it any more)
    srv = prdf.Server(slots=slots)
    for h in hs:
        srv.add(h)
    hs[0].close()
    srv.close()
    assert hs[1].tuning().blocks_per_sm == before[1]
    hs[1].close()


@pytest.mark.parametrize("slots", [1, 2, 3])
def test_bounded_runs_give_the_same_ranks(env, slots):
    # 16 M edges: runs of at most 32 iterations in a server of several slots, for requests alone and
    # for several in flight; 64-bit ranks do not depend on them
    prdf, torch = env
    gs = [synth.rmat(s, 16, seed=15 + s) for s in (20, 17, 14)]
    bs = [synth.BatchStream(g, seed=16) for g in gs]
    batches = [[b.next(f) for f in (1e-4, 1e-3, 1e-5, 1e-4)] for b in bs]
    streams = [torch.cuda.Stream() for _ in gs]
    made = [[prdf.Graph(g.n, g.src, g.dst, None, s.cuda_stream) for g, s in zip(gs, streams)] for _ in range(2)]
    for hs in made:
        for h in hs:
            h.static()
    want = []
    for h, todo in zip(made[0], batches):
        want.append([])
        for b in todo:
            h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
            st = h.frontier()
            want[-1].append((st.iterations, st.converged, st.affected_final))
    with prdf.Server(slots=slots, max_coalesce=1, hbm_reserve_bytes=0) as srv:
        idx = [srv.add(h) for h in made[1]]

        def submit(i, k):
            b = batches[i][k]
            return srv.submit(idx[i], b.del_src, b.del_dst, b.ins_src, b.ins_dst)

        got = [[] for _ in gs]
        for k, together in enumerate((False, True, False, True)):
            tickets = []
            for i in range(len(gs)):
                tickets.append(submit(i, k))
                if not together:
                    srv.wait(tickets[-1])
            for i, t in enumerate(tickets):
                r = srv.wait(t)
                assert r.status == prdf.PR_OK
                got[i].append((r.stats.iterations, r.stats.converged, r.stats.affected_final))
    assert got == want
    assert max(x[0] for x in want[0]) > 32
    for a, b in zip(*made):
        assert np.array_equal(a.ranks(), b.ranks())
        a.close()
        b.close()
