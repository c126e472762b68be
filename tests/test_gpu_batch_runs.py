"""Batched handles: the iterations in one launch of their own (df_split 1) against the one
persistent launch (df_split 0).

Both sum every row in the same order, so ranks, per-graph iterations and L-inf changes, and
affected sets agree bit for bit in both precisions: over graphs of one vertex up to graphs
larger than an SM's shared copy of contributions, more graphs than blocks, graphs without
edges, iteration limits (a graph's last iteration still marks), and every kind of call, with
and without graph replay.
"""
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


def _path(n):
    return synth.from_pairs(n, [(i, i + 1) for i in range(n - 1)], f"path-{n}")


def _set(name):
    if name == "large":  # larger than the copies (32 K vertices FP32, 16 K in 64-bit mode), among small ones
        return [_path(3), synth.rmat(16, 8, seed=1), synth.rmat(11, 4, seed=2), synth.rmat(15, 8, seed=3), _path(2)]
    if name == "many":
        rng = np.random.default_rng(3)
        gs = [synth.from_pairs(int(n), [], "empty") if n % 3 == 0 else _path(int(n)) for n in rng.integers(1, 40, 330)]
        return gs + [synth.rmat(int(s), 6, seed=int(9 + s)) for s in rng.integers(4, 10, 30)]
    assert name == "hubs"  # rows of several chunks; a chain on which marks travel for many iterations
    star = synth.from_pairs(5000, [(i, 0) for i in range(1, 5000)] + [(0, i) for i in range(1, 5000, 7)], "star")
    return [star, _path(300), synth.rmat(13, 16, seed=4), synth.from_pairs(1, [], "one")]


def _cat(gs, parts):
    first = np.cumsum([0] + [g.n for g in gs])
    return [np.concatenate([p[k].astype(np.uint64) + first[i] for i, p in enumerate(parts)]).astype(np.uint32)
            if parts else np.zeros(0, np.uint32) for k in range(len(parts[0]))]


def _handle(prdf, gs, split, f32, max_iter, replay):
    src, dst = _cat(gs, [(g.src, g.dst) for g in gs])
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if f32 else prdf.PR_F64
    p.max_iter = max_iter
    h = prdf.Graph.batched([g.n for g in gs], src, dst, p)
    t = h.tuning()
    h.set_tuning(t.bin_lo, t.bin_hi, t.dense_div, t.blocks_per_sm, split)
    h.set_graph_launch(replay)
    return h


def _batches(gs, frac, seed):
    out = []
    for i, g in enumerate(gs):
        if g.m < 20:
            z = np.zeros(0, np.uint32)
            out.append((z, z, z, z))
            continue
        b = synth.BatchStream(g, seed=seed + i).next(frac)
        out.append((b.del_src, b.del_dst, b.ins_src, b.ins_dst))
    return _cat(gs, out)


def _run(h, gs, batches):
    res = []

    def note(st, marked):
        cs = h.component_stats()
        res.append((h.ranks().copy(), st.iterations, st.converged, st.affected_final, st.vertices_processed,
                    st.edges_processed, [(c.iterations, c.converged, c.affected_final, c.last_delta) for c in cs],
                    np.sort(h.affected()).tolist() if marked else None))

    note(h.static(), False)
    for k, b in enumerate(batches):
        h.apply(*b)
        call = ("frontier", "traversal", "frontier", "naive")[k % 4]
        note(getattr(h, call)(), call != "naive")
    return res


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("max_iter,replay", [(500, False), (500, True), (3, False), (0, False)])
@pytest.mark.parametrize("name", ["large", "many", "hubs"])
def test_runs_equal_the_single_launch(prdf, name, max_iter, replay, f32):
    gs = _set(name)
    batches = [_batches(gs, f, 50 + k) for k, f in enumerate((2e-3, 1e-2, 5e-2, 1e-3))]
    out = []
    for split in (1, 0):
        with _handle(prdf, gs, split, f32, max_iter, replay) as h:
            out.append(_run(h, gs, batches))
    for k, (x, y) in enumerate(zip(*out)):
        assert np.array_equal(x[0], y[0]), k
        assert x[1:] == y[1:], k
