"""Updates of rows at the lengths and change counts where the merge changes: rows a warp takes
(up to 512 entries and 64 changes), rows in slices of 2048 entries, rows that are emptied,
moved or filled, in both directions; large updates, refused ones and sequences.  The
adjacencies and the effective changes' marks are the oracle's, and the sweeps read them."""
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


def _check(h, G):
    for d in (0, 1):
        o, c = h.csr(d)
        eo, ec = G.csr(d)
        assert np.array_equal(o, eo) and np.array_equal(c, ec)


def _u(a):
    return np.asarray(a, dtype=np.uint32)


def _hub_graph(length):
    """Out-hub 0 and in-hub 1 whose rows hold every second id, over a ring of all vertices."""
    n = 2 * length + 50
    v = np.arange(n, dtype=np.uint32)
    ids = _u(10 + 2 * np.arange(length - 2))
    src = np.concatenate([v, np.zeros(ids.size, np.uint32), ids])
    dst = np.concatenate([np.roll(v, -1), ids, np.ones(ids.size, np.uint32)])
    return n, src, dst, ids


def _update(n, ids, c, kind, rng):
    k_del = {"ins": 0, "del": c, "mix": c // 2}[kind]
    k_del = min(k_del, ids.size)
    k_ins = min(0 if kind == "del" else c - k_del, n - 30 - ids.size)
    out = np.sort(rng.choice(ids, k_del, replace=False))
    if k_del > 2:  # the ends of the row too
        out[0], out[-1] = ids[0], ids[-1]
    odd = _u(11 + 2 * np.arange((n - 20) // 2))
    into = rng.choice(odd[odd < n], min(k_ins, int((odd < n).sum())), replace=False)
    z, o = np.zeros, np.ones
    ds = np.concatenate([z(out.size), out])
    dd = np.concatenate([out, o(out.size)])
    is_ = np.concatenate([z(into.size), into])
    id_ = np.concatenate([into, o(into.size)])
    return _u(ds), _u(dd), _u(is_), _u(id_)


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("kind", ["ins", "del", "mix"])
@pytest.mark.parametrize("length", [3, 4, 511, 512, 513, 2047, 2048, 2049, 4096, 4097, 9001])
def test_row_lengths(prdf, length, kind, f32):
    rng = np.random.default_rng(length)
    n, src, dst, ids = _hub_graph(length)
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    p.vertex_order = 1  # in-rows in the caller's order, so that float sums are those of a fresh handle
    with prdf.Graph(n, src, dst, p) as h:
        G = oracle.Graph.build(n, src, dst)
        h.static()
        for c in (1, 63, 64, 65, 2048, 5000):
            up = _update(n, ids, c, kind, rng)
            R = h.ranks().copy()
            h.apply(*up)
            H, ed, ei = G.apply(*up)
            _check(h, H)
            st = h.frontier()
            if not f32 and ed[0].size + ei[0].size:
                # oracle sums of at most ~1e4 doubles: 1e4 2^-53 of a rank, over 1 / (1 - 0.85)
                ro, aff, so = oracle.df_sync(G, H, ed, ei, R)
                assert np.array_equal(np.sort(h.affected()), np.nonzero(aff)[0])
                assert np.abs(h.ranks() - ro).max() <= 1e-10 and st.iterations == so.iterations
            G = H
        h.static()
        s, d = _pairs(H)
        with prdf.Graph(n, s, d, p) as fresh:
            fresh.static()
            assert np.array_equal(h.ranks(), fresh.ranks())


def _pairs(G):
    o, c = G.csr(0)
    return _u(np.repeat(np.arange(o.size - 1), np.diff(o.astype(np.int64)))), _u(c)


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("total", [155647, 155648, 155649, (1 << 20) + 1])
def test_large_updates(prdf, total, f32):  # (152 blocks of 1024 pairs, and many rounds of them)
    g = synth.rmat(16, 8, seed=71)
    rng = np.random.default_rng(5)
    k = 50_000
    at = rng.choice(g.m, k, replace=False)
    is_, id_ = (rng.integers(0, g.n, total - k).astype(np.uint32) for _ in range(2))
    G = oracle.Graph.build(g.n, g.src, g.dst)
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    with prdf.Graph(g.n, g.src, g.dst, p) as h:
        h.apply(g.src[at], g.dst[at], is_, id_)
        H, _, _ = G.apply(g.src[at], g.dst[at], is_, id_)
        _check(h, H)


@pytest.mark.parametrize("k", [2048, 2049, 40000])
def test_refused_requests_leave_the_graph(prdf, k):
    g = synth.rmat(12, 8, seed=72)
    rng = np.random.default_rng(k)
    is_, id_ = (rng.integers(0, g.n, k).astype(np.uint32) for _ in range(2))
    bad = id_.copy()
    bad[k // 2] = g.n
    none = _u([])
    G = oracle.Graph.build(g.n, g.src, g.dst)
    with prdf.Graph(g.n, g.src, g.dst) as h:
        with pytest.raises(prdf.PrdfError):
            h.apply(none, none, is_, bad)
        _check(h, G)
        h.apply(none, none, is_, is_)  # self pairs only: nothing to do
        _check(h, G)
        h.apply(none, none, is_, id_)
        _check(h, G.apply(none, none, is_, id_)[0])


def test_batches_of_a_sequence(prdf):
    g = synth.rmat(13, 8, seed=73)
    G = oracle.Graph.build(g.n, g.src, g.dst)
    rng = np.random.default_rng(9)
    bs = []
    for size in (1, 30, 900, 1500, 0, 4000):
        at = rng.choice(g.m, size // 3, replace=False)
        is_, id_ = (rng.integers(0, g.n, size - size // 3).astype(np.uint32) for _ in range(2))
        bs.append((g.src[at], g.dst[at], is_, id_))
    with prdf.Graph(g.n, g.src, g.dst) as h:
        h.apply_batches(bs)
        for b in bs:
            G = G.apply(*b)[0]
        _check(h, G)
