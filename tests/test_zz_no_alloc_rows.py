"""pr_static_noalloc at the row lengths where its iteration kernel changes how it sums a row:
four lanes a row up to 16 in-edges, listed segments of 64 beyond, and blocks with more long
rows or segments than their lists hold (whose warps sum the rest)."""
import ctypes

import numpy as np
import pytest

import __graft_entry__

pytestmark = pytest.mark.gpu

# a row of k terms is off by at most k rounding errors of its sum, whatever the order, here
# and in the reference; the iterations damp what they inherit by alpha, so 1 / (1 - alpha) < 7
# covers their sum
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf

    prdf.load()
    return prdf, torch


def _rows(torch, lens, seed):
    """In-edge CSR with the given row lengths; every vertex is a source at least once."""
    n = lens.numel()
    lens = torch.clamp(lens, min=1)
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(lens, 0)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    col = torch.randint(0, n, (int(off[-1]),), generator=gen, device="cuda", dtype=torch.int64)
    col[off[:-1]] = torch.randperm(n, generator=gen, device="cuda")
    return off, col.to(torch.int32)


def _reference(torch, off, col, n, iters):
    deg = torch.bincount(col.to(torch.int64), minlength=n).to(torch.float64)
    row = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    src = col.to(torch.int64)
    r = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    for _ in range(iters):
        r = 0.15 / n + 0.85 * torch.zeros_like(r).index_add_(0, row, (r / deg)[src])
    return r


def _lens(torch, name):
    t = lambda x: torch.as_tensor(x, dtype=torch.int64, device="cuda")  # noqa: E731
    if name == "one":
        return t([1])
    if name == "few":
        return t([1, 33, 2, 513, 31])
    if name == "edges":
        return t(([1, 7, 8, 15, 16, 17, 32, 33, 63, 64, 65, 96, 127, 128, 129, 511, 1025, 4097] * 120)[:2053])
    if name == "hub":
        x = np.ones(30011, np.int64)
        x[::7] = 40
        x[12345] = 200003  # more than 1024 segments of 64 edges
        x[12346] = 65537
        return t(x)
    if name == "long-rows":  # more than 1024 long rows a block
        return t(np.where(np.arange(200003) % 5 == 0, 20, 130 + np.arange(200003) % 97))
    assert name == "segments"  # more than 2048 segments a block
    return t(np.full(24001, 6700))


@pytest.mark.parametrize("name", ["one", "few", "edges", "hub", "long-rows", "segments"])
@pytest.mark.parametrize("iters", [0, 1, 4])
def test_rows(env, name, iters):
    prdf, torch = env
    lens = _lens(torch, name)
    n = lens.numel()
    off, col = _rows(torch, lens, 5)
    p = prdf.pr_params_default()
    p.max_iter = iters
    p.tol = 0.0
    outs = []
    for _ in range(2):
        out = torch.full((n,), -1.0, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        st = prdf.pr_static_noalloc(n, off, col, out, params=p, stream=torch.cuda.current_stream().cuda_stream)
        outs.append(out)
    ref = _reference(torch, off, col, n, iters)
    rel = float(((outs[0] - ref).abs() / ref).max())
    assert rel <= 2 * 7 * (int(lens.max()) + 8) * EPS, (name, rel)
    assert torch.equal(outs[0], outs[1])  # one order of additions
    # a single vertex is at its fixed point at once; nothing else here converges exactly
    assert st.iterations == (min(iters, 1) if n == 1 else iters)


def test_stop_is_the_linf_change(env):
    prdf, torch = env
    off, col = _rows(torch, _lens(torch, "edges"), 9)
    n = off.numel() - 1
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    st = prdf.pr_static_noalloc(n, off, col, out, stream=torch.cuda.current_stream().cuda_stream)
    a, b = (_reference(torch, off, col, n, k) for k in (st.iterations - 1, st.iterations))
    assert st.converged and st.last_delta <= 1e-10
    assert abs(float((b - a).abs().max()) - st.last_delta) <= 1e-15
    c = _reference(torch, off, col, n, st.iterations - 2)
    assert float((a - c).abs().max()) > 1e-10 - 1e-15
