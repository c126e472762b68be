"""The asynchronous form reads, in an iteration, ranks updated earlier in the same iteration,
the hubs' too.

8192 hubs with 128 leaves each: leaf <- its hub, hub <- the leaves of the hub before.  The long rows
(hubs) are swept first, so most leaves are reached after their hub's new value is out.  After one
iteration over all vertices a leaf's rank is the synchronous one (from its hub's old value) or
clearly below it (from the new one).  With every hub's value copied at the start of the
iteration all would be synchronous.  The copies of whole graphs (at most 16 K vertices) take the same
path; there the results are only held to the synchronous form's."""
import numpy as np
import pytest

import __graft_entry__
import synth

pytestmark = pytest.mark.gpu

HUBS, PER = 8192, 128


@pytest.fixture(scope="module")
def prdf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf as mod

    mod.load()
    return mod


@pytest.mark.parametrize("f32", [False, True])
def test_leaves_see_their_hubs_new_ranks(prdf, f32):
    n = HUBS * (PER + 1)
    hub = np.arange(HUBS, dtype=np.uint32)
    leaf = np.arange(HUBS, n, dtype=np.uint32)
    mine = np.repeat(hub, PER)
    src = np.concatenate([mine, leaf])
    dst = np.concatenate([leaf, (mine + 1) % HUBS]).astype(np.uint32)
    p = prdf.pr_params_default()
    p.vertex_order = 2
    p.max_iter = 1
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    R = np.full(n, 0.5 / leaf.size)
    R[:HUBS] = 0.5 / HUBS
    none = np.zeros(0, np.uint32)
    got = []
    for call in ("frontier", "frontier_async"):
        with prdf.Graph(n, src, dst, p) as h:
            h.set_ranks(R)
            h.apply(none, none, hub, (hub + 7) % HUBS)  # every hub a source: all vertices affected
            st = getattr(h, call)()
            assert st.iterations == 1 and st.affected_final == n
            got.append(h.ranks().copy())
    sync, asy = got
    base, a, out = 0.15 / n, 0.85, PER + 2  # hubs: leaves, the new edge, the self-loop
    new = base + a * (R[:HUBS] / out + R[(hub + HUBS - 7) % HUBS] / out + PER * R[HUBS] / 2)
    # FP32: 130 terms of a hub's sum, half an ulp (2^-24) each of at most the sum; 64-bit: 2^-62
    # a term and the oracle's own doubles
    tol = 130 * 2.0 ** -24 * new.max() if f32 else 1e-15
    assert np.abs(sync[:HUBS] - new).max() <= tol
    old_leaf = base + a * (R[HUBS] / 2 + R[0] / out)
    # an updated hub has at most its old leaves' and the old hub's largest values in its sum
    top_leaf = base + a * (R[HUBS] / 2 + (base + a * (2 * R[0] / out + PER * old_leaf / 2)) / out)
    small = tol / out + (4 * 2.0 ** -24 * old_leaf if f32 else 1e-15)
    assert old_leaf - top_leaf > 100 * small
    assert np.abs(sync[HUBS:] - old_leaf).max() <= small
    leaves = asy[HUBS:]
    is_old = np.abs(leaves - old_leaf) <= small
    is_new = (leaves <= top_leaf + small) & (leaves >= base + a * R[HUBS] / 2 - small)
    assert np.all(is_old | is_new)
    assert is_new.mean() >= 0.25, is_new.mean()


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("scale", [9, 13, 16])
def test_agrees_with_the_synchronous_form(prdf, scale, f32):
    g = synth.rmat(scale, 8, seed=60 + scale)
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    bs = synth.BatchStream(g, seed=61)
    with prdf.Graph(g.n, g.src, g.dst, p) as h, prdf.Graph(g.n, g.src, g.dst, p) as s:
        s.static()
        for frac in (1e-2, 1e-3, 5e-2):
            b = bs.next(frac)
            h.set_ranks(s.ranks())
            for x in (h, s):
                x.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
            st, st_s = h.frontier_async(), s.frontier()
            assert st.converged and st_s.converged
            # both stop at a change of tau = 1e-10: 2 tau / (1 - alpha) apart at most; FP32: its rounding
            assert np.abs(h.ranks() - s.ranks()).max() <= (1e-6 if f32 else 2e-9)
