"""Batched handles: what one call or one handle may leave behind for the next."""
import numpy as np
import pytest

import __graft_entry__
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


def _cat(gs):
    first = np.cumsum([0] + [g.n for g in gs])
    return [np.concatenate([np.asarray(getattr(g, k), np.uint32) + np.uint32(first[i]) for i, g in enumerate(gs)])
            for k in ("src", "dst")]


def test_traversal_without_iterations_leaves_no_marks(prdf):
    # every block must see the marking launch's status before the first one is done, and clears
    # the marks of its share of the vertices: the affected set of each call is that of its batch
    gs = [synth.rmat(16, 4, seed=3), synth.rmat(15, 4, seed=4)]
    src, dst = _cat(gs)
    n, m = sum(g.n for g in gs), src.size
    p = prdf.pr_params_default()
    p.max_iter = 0
    none = np.zeros(0, np.uint32)
    with prdf.Graph.batched([g.n for g in gs], src, dst, p) as h, prdf.Graph(n, src, dst, p) as one:
        for k in range(40):
            at = np.array([k * (m // 40)])
            back = (none, none) if k % 2 else (src[at], dst[at])
            out = (src[at], dst[at]) if k % 2 else (none, none)
            h.apply(*out, *back)
            one.apply(*out, *back)
            for x in (h, one):
                x.traversal()
            assert np.array_equal(np.sort(h.affected()), np.sort(one.affected())), k


def _batch(gs, k):
    """A few deleted edges of every graph that has some, spread by k."""
    first = np.cumsum([0] + [g.n for g in gs])
    at = [np.arange(k % 7, g.m, max(1, g.m // 9)) for g in gs]
    return [np.concatenate([np.asarray(getattr(g, c), np.uint32)[i] + np.uint32(f)
                            for g, i, f in zip(gs, at, first)]).astype(np.uint32) for c in ("src", "dst")]


@pytest.mark.parametrize("replay", [False, True])
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("order", [(150, 3), (3, 150), (150, 3, 2), (700, 3)])
def test_handles_of_different_graph_counts(prdf, order, f32, replay):
    # all alive at once; every one must give what it gives alone, whichever was made last
    none = np.zeros(0, np.uint32)
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64

    def make(c):
        gs = [synth.rmat(4 + (i + c) % 6, 4, seed=9 + i % 13) for i in range(c)]
        h = prdf.Graph.batched([g.n for g in gs], *_cat(gs), p)
        h.set_graph_launch(replay)
        return gs, h

    def calls(gs, h):
        out = [h.static().converged, h.ranks().copy()]
        for k, call in enumerate(("frontier", "naive", "traversal", "frontier")):
            d = _batch(gs, k)
            h.apply(*(d if k % 2 == 0 else (none, none)), *((none, none) if k % 2 == 0 else _batch(gs, k - 1)))
            st = getattr(h, call)()
            out += [st.iterations, st.converged, st.affected_final, h.ranks().copy()]
        return out

    alone = []
    for c in order:
        gs, h = make(c)
        with h:
            alone.append(calls(gs, h))
    made = [make(c) for c in order]
    for (gs, h), want in zip(made, alone):
        got = calls(gs, h)
        assert all(np.array_equal(x, y) for x, y in zip(got, want))
    for _, h in made:
        h.close()


@pytest.mark.parametrize("f32", [False, True])
def test_calls_over_every_vertex(prdf, f32):
    # graphs large enough for a launch of their own (4 M edges, 4096 vertices on average), from one
    # vertex up to more than an SM's copy holds: bit for bit the one persistent launch, whatever
    # handle is made in between
    gs = [synth.rmat(17, 16, seed=3), synth.rmat(16, 16, seed=4), synth.from_pairs(1, [], "one"),
          synth.rmat(17, 16, seed=5), synth.rmat(11, 8, seed=6)]
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    out = []
    for split, max_iter in ((1, 500), (0, 500), (1, 3), (0, 3), (1, 0), (0, 0)):
        p.max_iter = max_iter
        with prdf.Graph.batched([g.n for g in gs], *_cat(gs), p) as h:
            assert h.info()[1] >= 4 << 20
            t = h.tuning()
            h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, split)
            with prdf.Graph.batched([2, 3], np.array([0], np.uint32), np.array([1], np.uint32), p) as small:
                small.static()
            res = []
            for k, call in enumerate(("static", "naive", "naive", "static")):
                st = getattr(h, call)()
                res.append((h.ranks().copy(), st.iterations, st.converged,
                            [(c.iterations, c.converged, c.last_delta) for c in h.component_stats()]))
                h.apply(*_batch(gs, k), np.zeros(0, np.uint32), np.zeros(0, np.uint32))
            out.append(res)
    for a, b in zip(out[::2], out[1::2]):
        for x, y in zip(a, b):
            assert np.array_equal(x[0], y[0]) and x[1:] == y[1:]
