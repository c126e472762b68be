"""Timed workloads of the Dynamic Frontier PageRank library, through its Python binding.

A case is a plain dict.  Kinds:

* ``update``    a graph kept on the device takes a batch of edge changes, its ranks are brought
                up to date and read; then the inverse batch, the same way.  One pass is thus
                two updates and leaves the edges as it found them.
* ``static``    ranks of a resident graph from 1/n, and their readout.
* ``snapshot``  an edge list on the device becomes a handle, is ranked, read and dropped.
* ``batched``   as ``update`` for a handle of many independent graphs, one launch for all.
* ``serve``     a request loop over several resident graphs serves two requests per graph.
* ``noalloc``   ranks of a caller's own in-edge CSR, without device allocations.

Graphs follow the repository's generators (R-MAT with a, b, c, d = 0.57, 0.19, 0.19, 0.05;
grids with 1% long-range arcs; symmetric chains like the k-mer graphs), drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2401_03256_gb300 import prdf

ALPHA, TOL, FTOL, MAX_ITER = 0.85, 1e-10, 1e-15, 500
DEV = "cuda"


def listed():
    rmat = {"kind": "update", "graph": "rmat", "method": "frontier", "dead_end": "selfloop"}
    return [
        # the plain method on a small graph: a dozen changed edges, bound by latency and launches
        {**rmat, "name": "update-rmat14-f64", "n": 1 << 14, "degree": 8.0, "frac": 1e-4, "precision": "f64"},
        # a social or web graph of ordinary size, a small batch (the benchmark's graph)
        {**rmat, "name": "update-rmat22-f64", "n": 1 << 22, "degree": 16.0, "frac": 1e-5, "precision": "f64"},
        # the largest power-law graph and the largest batch, single-precision ranks
        {**rmat, "name": "update-rmat24-f32", "n": 1 << 24, "degree": 16.0, "frac": 1e-3, "precision": "f32"},
        # a warm restart over all vertices after a large batch, vertex count not a power of two
        {**rmat, "name": "naive-rmat1.3M-f32", "n": 1300021, "degree": 16.0, "frac": 1e-3, "precision": "f32",
         "method": "naive"},
        # dead ends spread over all vertices instead of self-loops, odd vertex count
        {**rmat, "name": "teleport-rmat200K-f64", "n": 200003, "degree": 8.0, "frac": 1e-4, "precision": "f64",
         "dead_end": "teleport"},
        # a road network: high diameter, the frontier stays local
        {"name": "update-grid4900-f32", "kind": "update", "graph": "grid", "method": "frontier",
         "dead_end": "selfloop", "n": 4900 * 4900, "degree": 4.0, "frac": 1e-5, "precision": "f32"},
        # a low-degree k-mer graph, a batch whose frontier reaches a large part of it
        {"name": "update-kmer20M-f64", "kind": "update", "graph": "kmer", "method": "frontier",
         "dead_end": "selfloop", "n": 20000000, "degree": 2.1, "frac": 1e-4, "precision": "f64"},
        # all ranks of a resident graph from scratch
        {"name": "static-rmat22-f64", "kind": "static", "graph": "rmat", "dead_end": "selfloop", "n": 1 << 22,
         "degree": 16.0, "precision": "f64"},
        # a one-off ranking of an edge list: handle creation, ranking, readout
        {"name": "snapshot-rmat20-f64", "kind": "snapshot", "graph": "rmat", "dead_end": "selfloop", "n": 1 << 20,
         "degree": 16.0, "precision": "f64"},
        # many graphs of mixed sizes, each with a batch of its own, in one handle
        {"name": "batched-256-f32", "kind": "batched", "graphs": 256, "scale_lo": 10, "scale_hi": 18, "degree": 8.0,
         "precision": "f32"},
        # requests against several resident graphs, two on the device at a time
        {"name": "serve-5-f32", "kind": "serve", "graphs": 5, "scale_lo": 16, "scale_hi": 20, "degree": 16.0,
         "frac": 1e-5, "slots": 2, "precision": "f32"},
        # a caller that hands over its own CSR and must not allocate
        {"name": "noalloc-rmat60K-f64", "kind": "noalloc", "graph": "rmat", "dead_end": "selfloop", "n": 60013,
         "degree": 16.0, "precision": "f64"},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["update"] * 6 + ["static", "snapshot", "batched", "serve", "noalloc"])
    precision = rng.choice(["f64", "f32"])
    frac = 10.0 ** rng.uniform(-7.0, -3.0)
    if kind == "update":
        graph = rng.choice(["rmat", "rmat", "rmat", "grid", "kmer"])
        dead_end = rng.choice(["selfloop"] * 4 + ["teleport"])
        method = rng.choice(["frontier", "frontier", "frontier", "naive"])
        if graph == "rmat":
            hi = 1 << (20 if dead_end == "teleport" else 23)
            return {"kind": kind, "graph": graph, "method": method, "dead_end": dead_end, "n": log_int(1 << 12, hi),
                    "degree": rng.choice([4.0, 8.0, 16.0]), "frac": frac, "precision": precision}
        if graph == "grid":
            side = log_int(100, 4900)
            return {"kind": kind, "graph": graph, "method": method, "dead_end": "selfloop", "n": side * side,
                    "degree": 4.0, "frac": frac, "precision": precision}
        return {"kind": kind, "graph": graph, "method": method, "dead_end": "selfloop",
                "n": log_int(20000, 20000000), "degree": 2.1, "frac": frac, "precision": precision}
    if kind == "static":
        return {"kind": kind, "graph": "rmat", "dead_end": rng.choice(["selfloop"] * 3 + ["teleport"]),
                "n": log_int(1 << 12, 1 << 21), "degree": rng.choice([4.0, 8.0, 16.0]), "precision": precision}
    if kind == "snapshot":
        return {"kind": kind, "graph": "rmat", "dead_end": "selfloop", "n": log_int(1 << 12, 1 << 20),
                "degree": rng.choice([4.0, 8.0, 16.0]), "precision": precision}
    if kind == "batched":
        lo = rng.randint(8, 12)
        return {"kind": kind, "graphs": log_int(8, 256), "scale_lo": lo, "scale_hi": rng.randint(lo + 1, 17),
                "degree": 8.0, "precision": precision}
    if kind == "serve":
        lo = rng.randint(12, 16)
        return {"kind": kind, "graphs": rng.randint(3, 5), "scale_lo": lo, "scale_hi": rng.randint(lo + 1, 19),
                "degree": 16.0, "frac": frac, "slots": rng.choice([1, 2, 3]), "precision": precision}
    return {"kind": kind, "graph": "rmat", "dead_end": "selfloop", "n": log_int(1 << 9, 1 << 18),
            "degree": rng.choice([4.0, 8.0, 16.0]), "precision": "f64"}


# ---------------------------------------------------------------------------- inputs ----


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _rand(k, gen):
    return torch.rand(int(k), generator=gen, device=DEV)


def _randint(hi, k, gen):
    return torch.randint(0, int(hi), (int(k),), generator=gen, device=DEV, dtype=torch.int64)


def _rmat_pairs(scale, k, gen):
    """k R-MAT samples of 2^scale vertices (scale: an int, or a tensor of k ints)."""
    u = torch.zeros(k, dtype=torch.int64, device=DEV)
    v = torch.zeros(k, dtype=torch.int64, device=DEV)
    top = int(scale.max()) if torch.is_tensor(scale) else scale
    for level in range(top):
        r = _rand(k, gen)
        bu = r >= 0.76
        bv = ((r >= 0.57) & (r < 0.76)) | (r >= 0.95)
        if torch.is_tensor(scale):
            live = scale > level
            bu &= live
            bv &= live
        u += bu.to(torch.int64) << level
        v += bv.to(torch.int64) << level
    return u, v


def _edge_keys(case, gen):
    """Sorted distinct keys u * n + v of the graph's edges, without self-pairs."""
    n = case["n"]
    if case["graph"] == "rmat":
        scale = max(1, (n - 1).bit_length())
        label = torch.randperm(1 << scale, generator=gen, device=DEV)
        total, parts = int(round(case["degree"] * n)), []
        while total > 0:
            k = min(total, 1 << 26)
            u, v = _rmat_pairs(scale, k, gen)
            parts.append((label[u] % n) * n + label[v] % n)
            total -= k
        keys = torch.cat(parts)
    elif case["graph"] == "grid":
        side = math.isqrt(n)
        i = torch.arange(n, device=DEV)
        row, col = i // side, i % side
        parts = [i[col + 1 < side] * (n + 1) + 1, i[col > 0] * (n + 1) - 1,
                 i[row + 1 < side] * (n + 1) + side, i[row > 0] * (n + 1) - side,
                 _randint(n * n, max(1, n // 25), gen)]
        keys = torch.cat(parts)
    else:
        # symmetric chains over a random order: mean length 24, a cut end joining a vertex a
        # little further along, 5% more such short branches
        label = torch.randperm(n, generator=gen, device=DEV)
        i = torch.arange(n - 1, device=DEV)
        cut = _rand(n - 1, gen) < 1.0 / 24
        step = torch.where(cut, 2 + _randint(64, n - 1, gen), torch.ones_like(i))
        a, b = i, torch.clamp(i + step, max=n - 1)
        j = _randint(n, max(1, n // 20), gen)
        a, b = torch.cat([a, j]), torch.cat([b, torch.clamp(j + 2 + _randint(64, j.numel(), gen), max=n - 1)])
        a, b = label[a], label[b]
        keys = torch.cat([a * n + b, b * n + a])
    keys = keys[keys // n != keys % n]
    return torch.unique(keys)


def _batch_keys(keys, n, frac, gen):
    """Deleted and inserted keys: k = max(1, round(frac |E|)), 80% insertions of uniform absent pairs."""
    m = keys.numel()
    k = max(1, round(frac * m))
    k_ins = round(0.8 * k)
    cut = keys[torch.unique(_randint(m, k - k_ins, gen))]
    new = torch.unique(_randint(n * n, k_ins + 8, gen))
    new = new[new // n != new % n]
    at = torch.clamp(torch.searchsorted(keys, new), max=m - 1)
    new = new[keys[at] != new]
    return cut, new[torch.randperm(new.numel(), generator=gen, device=DEV)[:k_ins]]


def _ids(keys, n):
    return (keys // n).to(torch.int32), (keys % n).to(torch.int32)


def _host_batch(cut, new, n):
    """(del_src, del_dst, ins_src, ins_dst) host arrays, as requests arrive, and their inverse."""
    d = [x.cpu().numpy().view(np.uint32) for x in _ids(cut, n)]
    i = [x.cpu().numpy().view(np.uint32) for x in _ids(new, n)]
    return (d[0], d[1], i[0], i[1]), (i[0], i[1], d[0], d[1])


def _params(case):
    p = prdf.pr_params_default()
    p.precision = prdf.PR_F32 if case["precision"] == "f32" else prdf.PR_F64
    if case.get("dead_end") == "teleport":
        p.dead_end = prdf.PR_DEADEND_TELEPORT
    return p


def _single(case, seed):
    gen = _gen(seed)
    keys = _edge_keys(case, gen)
    cut, new = _batch_keys(keys, case["n"], case.get("frac", 1e-4), gen)
    return keys, cut, new


def _many(case, seed):
    """Graph sizes, edge keys (global ids, u * n + v), and a batch for every graph."""
    gen = _gen(seed)
    c = case["graphs"]
    # sizes spread evenly over the scales, in no order (the same for every seed)
    scale = case["scale_lo"] + 7 * torch.arange(c, device=DEV) % (case["scale_hi"] - case["scale_lo"] + 1)
    size = 1 << scale
    first = torch.cumsum(size, 0) - size
    n = int(size.sum())
    comp = torch.repeat_interleave(torch.arange(c, device=DEV), size)
    # a random relabelling inside every graph
    label = torch.argsort(comp.to(torch.float64) + _rand(n, gen).to(torch.float64) * 0.999)
    per = (case["degree"] * size).to(torch.int64)
    of = torch.repeat_interleave(torch.arange(c, device=DEV), per)
    u, v = _rmat_pairs(scale[of], of.numel(), gen)
    keys = label[first[of] + u] * n + label[first[of] + v]
    keys = torch.unique(keys[keys // n != keys % n])
    m_of = torch.bincount(comp[keys // n], minlength=c)
    start = torch.cumsum(m_of, 0) - m_of
    frac = torch.exp(_rand(c, gen).to(torch.float64) * math.log(100.0)) * 1e-4
    k = torch.clamp((frac * m_of).round().to(torch.int64), min=1)
    k_ins = (0.8 * k).round().to(torch.int64)
    d_of = torch.repeat_interleave(torch.arange(c, device=DEV), k - k_ins)
    cut = keys[torch.unique(start[d_of] + (_rand(d_of.numel(), gen).to(torch.float64) * m_of[d_of]).to(torch.int64))]
    i_of = torch.repeat_interleave(torch.arange(c, device=DEV), k_ins)
    a = first[i_of] + _randint(1 << 40, i_of.numel(), gen) % size[i_of]
    b = first[i_of] + _randint(1 << 40, i_of.numel(), gen) % size[i_of]
    new = torch.unique((a * n + b)[a != b])
    at = torch.clamp(torch.searchsorted(keys, new), max=keys.numel() - 1)
    return size, n, comp, keys, cut, new[keys[at] != new]


def _serve_cases(case):
    span = case["scale_hi"] - case["scale_lo"]
    return [{"kind": "update", "graph": "rmat", "dead_end": "selfloop", "degree": case["degree"],
             "frac": case["frac"] * 10.0 ** (k % 3 - 1), "precision": case["precision"],
             "n": 1 << (case["scale_lo"] + span * k // (case["graphs"] - 1))} for k in range(case["graphs"])]


def _in_csr(keys, n):
    """In-edge CSR (offsets, sources) of the edges u * n + v, self-loops added."""
    loops = torch.arange(n, device=DEV) * (n + 1)
    t = torch.sort((keys % n) * n + keys // n).values
    t = torch.sort(torch.cat([t, loops])).values
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(t // n, minlength=n), 0)
    return off, (t % n).to(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        graphs, batches, outs, streams = [], [], [], []
        for k, sub in enumerate(_serve_cases(case)):
            keys, cut, new = _single(sub, seed * 64 + k)
            src, dst = _ids(keys, sub["n"])
            torch.cuda.synchronize()
            streams.append(torch.cuda.Stream())
            g = prdf.Graph(sub["n"], src, dst, _params(sub), streams[-1].cuda_stream)
            g.static()
            graphs.append(g)
            batches.append(_host_batch(cut, new, sub["n"]))
            outs.append(torch.empty(sub["n"], dtype=torch.float64, device=DEV))
        return {"case": case, "graphs": graphs, "batches": batches, "outs": outs, "streams": streams}
    if kind == "batched":
        size, n, _, keys, cut, new = _many(case, seed)
        src, dst = _ids(keys, n)
        g = prdf.Graph.batched(size.tolist(), src, dst, _params(case))
        g.set_graph_launch(True)
        g.static()
        return {"case": case, "g": g, "batches": _host_batch(cut, new, n), "out": _outs(n, 2)}
    n = case["n"]
    keys, cut, new = _single(case, seed)
    if kind == "noalloc":
        off, col = _in_csr(keys, n)
        return {"case": case, "off": off, "col": col, "out": _outs(n, 1)}
    src, dst = _ids(keys, n)
    if kind == "snapshot":
        return {"case": case, "src": src, "dst": dst, "params": _params(case), "out": _outs(n, 1)}
    g = prdf.Graph(n, src, dst, _params(case))
    if kind == "update":
        g.static()
    return {"case": case, "g": g, "batches": _host_batch(cut, new, n), "out": _outs(n, 2)}


def _outs(n, k):
    return [torch.empty(n, dtype=torch.float64, device=DEV) for _ in range(k)]


def _read(case, ranks, stats=None):
    """What a program keeps of a rank call: the ranks in the precision it asked for, and in the
    64-bit mode (whose sums are exact in any order) the iterations and affected vertices."""
    if case["precision"] == "f32":
        return [ranks.to(torch.float32)]
    return [ranks] + ([int(stats.iterations), int(stats.affected_final)] if stats is not None else [])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("update", "batched"):
        g, got = s["g"], []
        for batch, out in zip(s["batches"], s["out"]):
            g.apply(*batch)
            st = g.naive() if case.get("method") == "naive" else g.frontier()
            got += _read(case, g.ranks(out), st)
        return got
    if kind == "static":
        st = s["g"].static()
        return _read(case, s["g"].ranks(s["out"][0]), st)
    if kind == "snapshot":
        with prdf.Graph(case["n"], s["src"], s["dst"], s["params"]) as g:
            st = g.static()
            return _read(case, g.ranks(s["out"][0]), st)
    if kind == "serve":
        # one rank call per request, so that every request has its own result
        with prdf.Server(slots=case["slots"], max_coalesce=1) as srv:
            at = [srv.add(g) for g in s["graphs"]]
            tickets = [srv.submit(gi, *b[k]) for k in range(2) for gi, b in zip(at, s["batches"])]
            for t in tickets:
                srv.wait(t)
        return [_read(case, g.ranks(out)) for g, out in zip(s["graphs"], s["outs"])]
    # the ranks alone: a change that meets the tolerance within rounding may take one more iteration
    prdf.pr_static_noalloc(case["n"], s["off"], s["col"], s["out"][0],
                           stream=torch.cuda.current_stream().cuda_stream)
    return _read(case, s["out"][0])


# ------------------------------------------------------------------------------ work ----


def work(case):
    """Every rank call reads the in-edges (4 bytes a column) and the old ranks once and writes
    the ranks it returns; a frontier that stays local (grids and chains, small batches) reads
    the batch and the old ranks and writes the ranks."""
    kind = case["kind"]
    es = 4 if case["precision"] == "f32" else 8
    if kind == "serve":
        parts = [work(c) for c in _serve_cases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "batched":
        lo, hi = case["scale_lo"], case["scale_hi"]
        n = case["graphs"] * ((2 << hi) - (1 << lo)) / (hi - lo + 1)
    else:
        n = case["n"]
    edges = n * (case["degree"] + 1)
    calls = 2 if kind in ("update", "batched") else 1
    pairs = case.get("frac", 1e-3) * edges if calls == 2 else 0
    if kind == "update" and case["graph"] != "rmat" and case["method"] == "frontier" and case["frac"] < 1e-3:
        edges = min(edges, 64 * pairs)
    if kind == "snapshot":
        return {"bytes": 8 * edges + (es + 8) * n, "flops": 2 * edges}
    return {"bytes": calls * (4 * edges + 8 * pairs + (es + 8) * n), "flops": 2 * calls * edges}


# ----------------------------------------------------------------------------- exact ----


class _Plain:
    """PageRank of one snapshot in float64: pull sums by a sparse product."""

    def __init__(self, keys, n, comp, size, teleport):
        self.n, self.teleport = n, teleport
        if not teleport:
            keys = torch.cat([keys, torch.arange(n, device=DEV) * (n + 1)])
        t = torch.sort((keys % n) * n + keys // n).values
        off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        off[1:] = torch.cumsum(torch.bincount(t // n, minlength=n), 0)
        self.A = torch.sparse_csr_tensor(off.to(torch.int32), (t % n).to(torch.int32),
                                         torch.ones(t.numel(), dtype=torch.float64, device=DEV), (n, n))
        self.deg = torch.bincount(keys // n, minlength=n).to(torch.float64)
        self.dead = self.deg == 0
        self.comp, self.size = comp, size.to(torch.float64)
        self.base = ((1.0 - ALPHA) / self.size)[comp]

    def dead_mass(self, r):
        return float(r[self.dead].sum()) if self.teleport else 0.0

    def sweep(self, r):
        c = torch.where(self.dead, torch.zeros_like(r), ALPHA * r / torch.clamp(self.deg, min=1.0))
        return self.base + self.A @ c + ALPHA * self.dead_mass(r) / self.n

    def change(self, r, q):
        out = torch.zeros(self.size.numel(), dtype=torch.float64, device=DEV)
        return out.scatter_reduce(0, self.comp, (r - q).abs(), "amax")

    def iterate(self, r, marked=None, d_prev=None):
        """All vertices (marked is None) or Algorithm 1 from the marked ones."""
        alive = torch.ones(self.size.numel(), dtype=torch.bool, device=DEV)
        for _ in range(MAX_ITER):
            go = alive[self.comp]
            if marked is not None:
                if self.teleport:
                    d = self.dead_mass(r)
                    if ALPHA * abs(d - d_prev) / self.n > FTOL:
                        marked = torch.ones_like(marked)
                    d_prev = d
                go = go & marked
            q = torch.where(go, self.sweep(r), r)
            if marked is not None:
                moved = ((q - r).abs() > FTOL).to(torch.float64)
                marked = marked | (self.A @ moved > 0)
            alive = alive & (self.change(q, r) > TOL)
            r = q
            if not bool(alive.any()):
                break
        return r

    def start(self):
        return self.iterate((1.0 / self.size)[self.comp])


def _apply(keys, cut, new):
    keep = torch.ones(keys.numel(), dtype=torch.bool, device=DEV)
    keep[torch.searchsorted(keys, cut)] = False
    return torch.sort(torch.cat([keys[keep], new])).values


def _two_updates(case, keys, cut, new, n, comp, size):
    teleport = case.get("dead_end") == "teleport"
    got = []
    G = _Plain(keys, n, comp, size, teleport)
    r = G.start()
    for dels, ins in ((cut, new), (new, cut)):
        d_prev = G.dead_mass(r)
        keys = _apply(keys, torch.sort(dels).values, ins)
        G = _Plain(keys, n, comp, size, teleport)
        marked = None
        if case.get("method") != "naive":
            src = torch.zeros(n, dtype=torch.float64, device=DEV)
            src[torch.cat([dels, ins]) // n] = 1.0
            marked = G.A @ src > 0
            marked[dels % n] = True
        r = G.iterate(r, marked, d_prev)
        got.append(r)
    return got


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return [[_two_updates(sub, *_single(sub, seed * 64 + k), sub["n"], *_one(sub["n"]))[1]]
                for k, sub in enumerate(_serve_cases(case))]
    if kind == "batched":
        size, n, comp, keys, cut, new = _many(case, seed)
        got = _two_updates(case, keys, cut, new, n, comp, size)
    elif kind == "update":
        got = _two_updates(case, *_single(case, seed), case["n"], *_one(case["n"]))
    else:
        keys, _, _ = _single(case, seed)
        got = [_Plain(keys, case["n"], *_one(case["n"]), case["dead_end"] == "teleport").start()]
    if case["precision"] == "f32" or kind == "noalloc":
        return got
    return [x for r in got for x in (r, None, None)]


def _one(n):
    return torch.zeros(n, dtype=torch.int64, device=DEV), torch.tensor([n], device=DEV)
