"""Runs of iterations in one launch, and contributions kept in shared memory.

Handles whose vertices of large out-degree come first in the internal numbering gather
those contributions from shared memory.  In 64-bit mode every sum is exact, so such a
handle must agree bit for bit with one that keeps the caller's numbering (no such vertices)
and with one that launches every iteration by itself (df_split 0), at sizes around a warp, a
block's rounds, a chunk, and the shared copy's capacity, through batch updates.  In FP32 the
order of a row's sum does not depend on the launches, so df_split 0 and 1 agree bit for bit
there too; updates keep the in-rows' order (the exported rows and ranks are the oracle's).
"""
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


def _star(n):
    """0 -> every vertex -> 0: one hub with in- and out-degree n - 1."""
    v = np.arange(1, n, dtype=np.uint32)
    z = np.zeros(n - 1, np.uint32)
    return synth.from_pairs(n, zip(np.concatenate([z, v]).tolist(), np.concatenate([v, z]).tolist()), f"star-{n}")


def _graph(name):
    kind, k = name.split("-")
    return _star(int(k)) if kind == "star" else synth.rmat(int(k), 8, seed=40 + int(k))


GRAPHS = ["star-2", "star-3", "star-5", "star-33", "star-513", "star-2000", "rmat-5", "rmat-9", "rmat-13", "rmat-16"]


def _handle(prdf, g, order, split, f32=False):
    p = prdf.pr_params_default()
    p.vertex_order = order
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    h = prdf.Graph(g.n, g.src, g.dst, p)
    t = h.tuning()
    h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, split)
    return h


def _batches(g):
    bs = synth.BatchStream(g, seed=17)
    return [bs.next(f) for f in (1e-3, 3e-2, 1e-2)], bs


def _run(h, batches):
    out = [h.static(), h.ranks().copy()]
    for k, b in enumerate(batches):
        h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
        st = (h.frontier, h.naive, h.traversal)[k % 3]()
        out += [st, h.ranks().copy(), np.sort(h.affected()) if k % 3 != 1 else np.zeros(0)]
    return out


def _same(a, b):
    for x, y in zip(a, b):
        if isinstance(x, np.ndarray):
            assert np.array_equal(x, y)
        else:
            assert (x.iterations, x.converged, x.affected_final, x.last_delta) == \
                (y.iterations, y.converged, y.affected_final, y.last_delta)


@pytest.mark.parametrize("name", GRAPHS)
def test_shared_copy_and_runs_are_invisible_fp64(prdf, name):
    g = _graph(name)
    batches = _batches(g)[0] if g.m > 60 else []
    got = []
    for order, split in ((2, 1), (1, 1), (2, 0)):
        with _handle(prdf, g, order, split) as h:
            got.append(_run(h, batches))
    _same(got[0], got[1])
    _same(got[0], got[2])


@pytest.mark.parametrize("name", GRAPHS)
def test_fp32_rows_keep_their_order(prdf, name):
    g = _graph(name)
    batches, bs = _batches(g) if g.m > 60 else ([], None)
    got = []
    for split in (1, 0):
        with _handle(prdf, g, 2, split, f32=True) as h:
            got.append(_run(h, batches))
            csr = [h.csr(d) for d in (0, 1)]
    # split 1: the dense iterations are sweeps, split 0: one persistent launch; same sums
    _same(got[0][:2], got[1][:2])
    if bs is None:
        return
    _same(got[0][2:4], got[1][2:4])
    c = bs.current()
    H = oracle.Graph.build(c.n, c.src, c.dst)
    for d in (0, 1):
        eo, ec = H.csr(d)
        assert np.array_equal(csr[d][0], eo) and np.array_equal(csr[d][1], ec)
    # FP32 ranks are held to the oracle's within 1e-6 after every kind of call
    assert np.max(np.abs(got[0][-2] - oracle.static_pr(H)[0])) <= 1e-6


def test_run_barrier_wait_runs_out_and_the_handle_recovers(prdf):
    # a limit of 1 us on the barrier waits: Static's run and a dense Dynamic Frontier call's end
    # early with PR_ERR_DEVICE_TIMEOUT, and the next calls start clean
    g = synth.rmat(14, 8, seed=31)
    b = synth.BatchStream(g, seed=3).next(1e-3)
    G = oracle.Graph.build(g.n, g.src, g.dst)
    R0, _ = oracle.static_pr(G)
    with _handle(prdf, g, 0, 1) as h:
        t = h.tuning()
        h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, 1, barrier_us=1)
        timed_out = 0
        for call in (h.static, h.static, h.frontier, h.static):
            try:
                call()
            except prdf.PrdfError as e:
                assert e.status == prdf.PR_ERR_DEVICE_TIMEOUT
                timed_out += 1
        assert timed_out > 0
        h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, 1, barrier_us=0)
        assert h.static().converged and np.max(np.abs(h.ranks() - R0)) <= 1e-9
        h.set_ranks(R0)
        h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
        H, ed, ei = G.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
        R_df, aff, _ = oracle.df_sync(G, H, ed, ei, R0)
        h.frontier()
        assert np.max(np.abs(h.ranks() - R_df)) <= 1e-9
