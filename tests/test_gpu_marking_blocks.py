"""The marking launch's two sizes (2 or 4 blocks an SM) around the line between them: calls of one
changed edge on a ring with a hub of many chunks, at 2^21 vertices and around, give the ranks
and affected sets of the one persistent launch bit for bit."""
import numpy as np
import pytest

import __graft_entry__

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hub", [False, True])
@pytest.mark.parametrize("n", [(1 << 21) - 1, 1 << 21, (1 << 21) + 1])
def test_few_marks(n, hub):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf

    prdf.load()
    v = np.arange(n, dtype=np.uint32)
    src, dst = v, np.roll(v, -1)
    if hub:  # every vertex points at vertex 7: a row of n entries, which passes its rank to one vertex
        src, dst = np.concatenate([src, v]), np.concatenate([dst, np.full(n, 7, np.uint32)])
    none = np.zeros(0, np.uint32)
    e = np.array([n // 2], np.uint32)
    out = []
    for split in (1, 0):
        with prdf.Graph(n, src, dst) as h:
            t = h.tuning()
            h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, split)
            h.static()
            res = [h.ranks().copy()]
            for up in ((none, none, e, e // 3), (e, e // 3, none, none)):
                h.apply(*up)
                for call in ("frontier", "traversal"):
                    st = getattr(h, call)()
                    res += [h.ranks().copy(), np.sort(h.affected()), np.array([st.iterations, st.affected_final])]
            out.append(res)
    assert all(np.array_equal(a, b) for a, b in zip(*out))
