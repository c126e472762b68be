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


@pytest.mark.parametrize("f32", [False, True])
def test_rows_repacked_without_a_change_of_tier(prdf, f32):
    # in-rows of 21 entries (28 slots) grow to 31 (64 slots), 200 an update: the second one finds
    # 1200 of 70,000 words left, so all rows are laid out anew, most of them elsewhere, and none
    # changes its tier; the sweeps must follow
    n = 2000
    v = np.arange(n)
    src = _u((np.repeat(v, 20) + np.tile(np.arange(1, 21), n)) % n)
    dst = _u(np.repeat(v, 20))
    G = oracle.Graph.build(n, src, dst)
    p = prdf.pr_params_default()
    p.vertex_order = 1
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    none = _u([])
    with prdf.Graph(n, src, dst, p) as h:
        h.static()
        for lo in (0, 1000, 200, 1200):
            rows = np.repeat(np.arange(lo, lo + 200), 10)
            up = (none, none, _u((rows + 100 + 37 * np.tile(np.arange(10), 200)) % n), _u(rows))
            h.apply(*up)
            G = G.apply(*up)[0]
            _check(h, G)
            ref = oracle.static_pr(G)[0]
            for call in ("frontier", "static"):
                getattr(h, call)()
                # a change of 1e-10 stops both: 2 tau / (1 - alpha) apart at most; FP32: its rounding
                assert np.abs(h.ranks() - ref).max() <= (1e-6 if f32 else 2e-9)


def _ring(n, k):
    v = np.arange(n)
    return _u((np.repeat(v, k) + np.tile(np.arange(1, k + 1), n)) % n), _u(np.repeat(v, k))


def _more(lo, rows, k, at):
    """k new in-edges for each of the rows from lo on, from vertices at, at + 37, ... further."""
    r = np.repeat(np.arange(lo, lo + rows), k)
    none = _u([])
    return none, none, _u((r + at + 37 * np.tile(np.arange(k), rows)) % 2000), _u(r)


def test_a_repack_without_room_leaves_the_rows_their_slots(prdf):
    # rows 400 to 409 fill their 28 slots; the update after the next needs a repack, whose allocation
    # fails; then the full rows must move, not grow over their neighbours
    src, dst = _ring(2000, 20)
    G = oracle.Graph.build(2000, src, dst)
    p = prdf.pr_params_default()
    p.vertex_order = 1
    with prdf.Graph(2000, src, dst, p) as h:
        for up in (_more(400, 10, 7, 500), _more(0, 200, 10, 100)):
            h.apply(*up)
            G = G.apply(*up)[0]
        big = _more(1000, 200, 10, 100)
        prdf.pr_inject_alloc_failure(0)
        try:
            with pytest.raises(prdf.PrdfError) as e:
                h.apply(*big)
        finally:
            prdf.pr_inject_alloc_failure(-1)
        assert e.value.status == prdf.PR_ERR_OUT_OF_MEMORY
        _check(h, G)
        for up in (_more(400, 10, 1, 900), big, _more(400, 10, 9, 1100)):
            h.apply(*up)
            G = G.apply(*up)[0]
            _check(h, G)
        h.static()
        assert np.abs(h.ranks() - oracle.static_pr(G)[0]).max() <= 2e-9


def test_no_room_for_the_sweep_items(prdf):
    # 32-edge chunks and no other tiers: the update takes every row from 21 entries to 33, so the
    # items outgrow their arrays.  Whichever allocation fails, a call that fails leaves the
    # graph as it was, one that does not has updated it, and both leave a usable handle
    src, dst = _ring(2000, 20)
    G = oracle.Graph.build(2000, src, dst)
    p = prdf.pr_params_default()
    p.vertex_order = 1
    big = _more(0, 2000, 12, 100)
    H = G.apply(*big)[0]
    failed = []
    for allowed in range(5):
        with prdf.Graph(2000, src, dst, p) as h:
            t = h.tuning()
            h.set_tuning(1, t.bin_hi, t.dense_div, t.blocks_per_sm, 1, 0, 32, 0)
            h.apply(*(_u([]), _u([]), big[3], big[3]))  # (self pairs: scratch for the real one)
            prdf.pr_inject_alloc_failure(allowed)
            try:
                h.apply(*big)
                now, ok = H, True
            except prdf.PrdfError as e:
                assert e.status == prdf.PR_ERR_OUT_OF_MEMORY
                now, ok = G, False
            finally:
                prdf.pr_inject_alloc_failure(-1)
            failed.append(not ok)
            _check(h, now)
            for up in (_more(5, 3, 2, 700), big):
                h.apply(*up)
                now = now.apply(*up)[0]
                _check(h, now)
            for call in ("frontier", "static"):
                getattr(h, call)()
                assert np.abs(h.ranks() - oracle.static_pr(now)[0]).max() <= 2e-9
    assert failed[0] and not failed[-1]


def test_a_rank_call_without_room_for_the_sweep_items(prdf):
    src, dst = _ring(2000, 20)
    G = oracle.Graph.build(2000, src, dst)
    p = prdf.pr_params_default()
    p.vertex_order = 1
    big, small = _more(0, 2000, 12, 100), _more(5, 3, 2, 700)
    with prdf.Graph(2000, src, dst, p) as h:
        t = h.tuning()
        h.set_tuning(1, t.bin_hi, t.dense_div, t.blocks_per_sm, 1, 0, 32, 0)
        h.apply(*(_u([]), _u([]), big[3], big[3]))
        prdf.pr_inject_alloc_failure(2)  # both adjacencies' new slots, not the items
        try:
            h.apply(*big)
            for call in (h.static, h.frontier, h.naive):
                with pytest.raises(prdf.PrdfError) as e:
                    call()
                assert e.value.status == prdf.PR_ERR_OUT_OF_MEMORY
            h.apply(*small)  # in the rows' own slots
        finally:
            prdf.pr_inject_alloc_failure(-1)
        G = G.apply(*big)[0].apply(*small)[0]
        _check(h, G)
        h.frontier()
        assert np.abs(h.ranks() - oracle.static_pr(G)[0]).max() <= 2e-9


@pytest.mark.parametrize("k", [2049, 5000, 200000])
def test_a_barrier_wait_of_the_plan_runs_out(prdf, k):
    # (updates of at most 2048 pairs are planned by one block, which waits for no other)
    n = 40000
    src, dst = _u(np.arange(n)), _u((np.arange(n) + 1) % n)
    rng = np.random.default_rng(k)
    none = _u([])
    G = oracle.Graph.build(n, src, dst)
    with prdf.Graph(n, src, dst) as h:
        t = h.tuning()
        ended = 0
        for _ in range(6):
            up = (none, none, *(rng.integers(0, n, k).astype(np.uint32) for _ in range(2)))
            h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, 1, 1)  # 1 us
            try:
                h.apply(*up)
                G = G.apply(*up)[0]
            except prdf.PrdfError as e:
                assert e.status == prdf.PR_ERR_DEVICE_TIMEOUT
                ended += 1
                _check(h, G)
                h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, 1, 0)
                h.apply(*up)
                G = G.apply(*up)[0]
            _check(h, G)
        assert ended > 0 or k < 200000  # a few blocks may always meet within the limit
        h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, 1, 0)
        h.frontier()
        assert np.abs(h.ranks() - oracle.static_pr(G)[0]).max() <= 2e-9
