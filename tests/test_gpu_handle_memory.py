"""A destroyed handle gives its device memory back, the device-side loops' too."""
import pytest

import __graft_entry__
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["static", "frontier", "frontier_async", "traversal"])
def test_destroyed_handles_leave_nothing(call):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf

    prdf.load()
    g = synth.rmat(13, 8, seed=1)
    b = synth.BatchStream(g, seed=2).next(5e-2)

    def one():
        with prdf.Graph(g.n, g.src, g.dst) as h:
            h.static()
            h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
            getattr(h, call)()

    for _ in range(5):
        one()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(60):
        one()
    # a loop takes 0.9 MB; the driver hands memory out 2 MB at a time
    assert free - torch.cuda.mem_get_info()[0] <= 8 << 20


@pytest.mark.parametrize("order", [1, 2])
def test_affected_sets_of_any_length_and_capacity(order):
    # short ones come through pinned memory (up to 16,384 ids), longer ones from the device, from up to
    # three lists, whole or cut at the caller's capacity
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    import ctypes

    import numpy as np
    import oracle
    from paper_2401_03256_gb300 import prdf

    lib = prdf.load()
    seen = set()
    for scale, frac, split in ((6, 1e-2, 1), (12, 1e-3, 0), (15, 1e-3, 1), (15, 1e-2, 0)):
        g = synth.rmat(scale, 8, seed=scale)
        G = oracle.Graph.build(g.n, g.src, g.dst)
        R, _ = oracle.static_pr(G)
        b = synth.BatchStream(g, seed=3).next(frac)
        p = prdf.pr_params_default()
        p.vertex_order = order
        p.max_iter = 1
        with prdf.Graph(g.n, g.src, g.dst, p) as h:
            t = h.tuning()
            h.set_tuning(1, 8, t.dense_div if split else 1, t.blocks_per_sm, split)
            h.set_ranks(R)
            h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
            H, ed, ei = G.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
            h.frontier()
            _, aff, _ = oracle.df_sync(G, H, ed, ei, R, oracle.Params(max_iter=1))
            want = np.nonzero(aff)[0]
            got = h.affected()
            assert np.array_equal(np.sort(got), want)
            seen.add(want.size > 16384)
            for cap in (0, 1, want.size // 2, want.size - 1, want.size + 5):
                out = np.full(want.size + 8, 7, np.uint32)
                cnt = ctypes.c_int64()
                assert lib.pr_get_affected(h.h, out.ctypes.data, cap, ctypes.byref(cnt)) == prdf.PR_OK
                k = min(cap, want.size)
                assert cnt.value == want.size and np.array_equal(out[:k], got[:k]) and np.all(out[k:] == 7)
    assert seen == {False, True}
