"""The autotuner leaves the marking launch's blocks per SM alone where what it times, Naive-dynamic
sweeps, runs in launches of other sizes."""
import pytest

import __graft_entry__
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["single", "batched", "batched, small", "teleport", "batched, one launch"])
def test_blocks_that_the_sweeps_do_not_use(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf

    prdf.load()
    # (batched handles of less than 4 M edges sweep every vertex in the persistent launch)
    g = synth.rmat(18, 16, seed=5) if kind == "batched" else synth.rmat(11, 8, seed=5)
    p = prdf.pr_params_default()
    if kind == "teleport":
        p.dead_end = prdf.PR_DEADEND_TELEPORT
    h = prdf.Graph.batched([g.n, 5], g.src, g.dst, p) if "batched" in kind else prdf.Graph(g.n, g.src, g.dst, p)
    with h:
        t = h.tuning()
        most = t.blocks_per_sm
        h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, 1, 0 if "one launch" in kind else 1)
        h.static()
        got = h.autotune(4).blocks_per_sm
        if kind in ("single", "batched"):
            assert got == 1
        else:  # the persistent launch: the largest sizes are tried
            assert max(1, most - 2) <= got <= most
        assert h.tuning().blocks_per_sm == got
