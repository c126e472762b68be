"""Graph creation and updates at the sizes where the sorts and searches change: key counts
around a block's sort, a radix tile and the switch between tile sizes, and rows around the
length from which the vertex numbering's search takes them in segments.  The exported
adjacencies are the oracle's, and ranks do not depend on the internal numbering."""
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


def _pairs(n, m, seed):
    rng = np.random.default_rng(seed)
    k = rng.choice(n * n, m, replace=False).astype(np.uint64)
    return (k // np.uint64(n)).astype(np.uint32), (k % np.uint64(n)).astype(np.uint32)


def _check(h, G):
    for d in (0, 1):
        o, c = h.csr(d)
        eo, ec = G.csr(d)
        assert np.array_equal(o, eo) and np.array_equal(c, ec)


# keys = pairs + vertices (self-loops): block sorts end at 4096 keys, radix tiles hold 1024
@pytest.mark.parametrize("m", [1, 3995, 3996, 3997, 5019, 5020, 5021, 9000])
@pytest.mark.parametrize("f32", [False, True])
def test_build_at_sort_sizes(prdf, m, f32):
    n = 100
    src, dst = _pairs(n, m, m)
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    with prdf.Graph(n, src, dst, p) as h:
        _check(h, oracle.Graph.build(n, src, dst))


@pytest.mark.parametrize("extra", [-1, 0, 1])
def test_build_at_the_switch_of_tile_sizes(prdf, extra):
    n = 3000
    src, dst = _pairs(n, 2_500_000 - n + extra, 7)
    with prdf.Graph(n, src, dst) as h:
        _check(h, oracle.Graph.build(n, src, dst))


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("k", [2047, 2048, 2049, 3071, 3072, 3073, 4096, 4097, 20000])
def test_update_at_sort_sizes(prdf, k, f32):
    g = synth.rmat(13, 8, seed=70)
    rng = np.random.default_rng(k)
    at = rng.choice(g.m, k // 3, replace=False)
    ds, dd = g.src[at], g.dst[at]
    is_, id_ = (rng.integers(0, g.n, k - k // 3).astype(np.uint32) for _ in range(2))
    G = oracle.Graph.build(g.n, g.src, g.dst)
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    with prdf.Graph(g.n, g.src, g.dst, p) as h:
        h.apply(ds, dd, is_, id_)
        H, _, _ = G.apply(ds, dd, is_, id_)
        _check(h, H)


@pytest.mark.parametrize("k", [1022, 1023, 1024, 1025, 1280, 1281, 5000])
def test_numbering_of_long_rows(prdf, k):
    # hubs with rows of k entries and their self-loop, in both directions
    n = k + 40
    v = np.arange(40, n, dtype=np.uint32)
    hubs = [np.full(k, h, np.uint32) for h in range(3)]
    src = np.concatenate(hubs[:2] + [v, v[: k // 2]])
    dst = np.concatenate([v, v, hubs[2], np.arange(3, 3 + k // 2, dtype=np.uint32) % 40])
    out = []
    for order in (1, 2, 3):
        p = prdf.pr_params_default()
        p.vertex_order = order
        with prdf.Graph(n, src, dst, p) as h:
            st = h.static()
            _check(h, oracle.Graph.build(n, src, dst))
            out.append((st.iterations, h.ranks().copy()))
    for it, r in out[1:]:
        assert it == out[0][0] and np.array_equal(r, out[0][1])
