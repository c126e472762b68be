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
