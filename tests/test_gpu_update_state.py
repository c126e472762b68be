"""Updates and what they leave behind: pending sources, the handle's sweep items and slots, on
every path an update can take, a failed allocation's among them."""
import numpy as np
import pytest

import __graft_entry__
import oracle

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


def _check(h, G):
    for d in (0, 1):
        o, c = h.csr(d)
        eo, ec = G.csr(d)
        assert np.array_equal(o, eo) and np.array_equal(c, ec)


def _u(a):
    return np.asarray(a, dtype=np.uint32)


@pytest.mark.parametrize("call", ["frontier", "traversal"])
@pytest.mark.parametrize("degree", [127, 128, 129, 190])
def test_a_row_updated_more_often_than_there_are_vertices(prdf, degree, call):
    # every update leaves its source pending; rows of more than 128 out-edges are queued for each
    n = 200
    src = np.concatenate([np.zeros(degree - 1, np.uint32), _u(np.arange(n))])
    dst = np.concatenate([_u(np.arange(1, degree)), _u((np.arange(n) + 1) % n)])
    G = oracle.Graph.build(n, src, dst)
    R, _ = oracle.static_pr(G)
    none, zero = _u([]), _u([0])
    with prdf.Graph(n, src, dst) as h:
        h.set_ranks(R)
        for k in range(2 * n + 1):
            e = (zero, _u([199 - k % 4]))
            up = (*e, none, none) if (k // 4) % 2 else (none, none, *e)
            h.apply(*up)
        H = G.apply(none, none, zero, _u([199]))[0]  # what the toggles leave
        _check(h, H)
        getattr(h, call)()
        ref = oracle.static_pr(H)[0]
        assert np.abs(h.ranks() - ref).max() <= 2e-9  # both stop at a change of 1e-10: 2 tau / (1 - alpha)
