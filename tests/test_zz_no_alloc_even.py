"""pr_static_noalloc on graphs whose rows are alike (a thread takes a row there): row lengths around
the limits of the split, with and without hubs, against 64-bit sums in numpy."""
import numpy as np
import pytest

import __graft_entry__

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hubs", [0, 1, 40])
@pytest.mark.parametrize("n,length", [(700, 1), (5000, 2), (5000, 5), (5000, 6), (5000, 7), (5000, 16), (5000, 17),
                                      (30000, 24), (5000, 64), (5000, 65), (3000, 255), (3000, 257), (200, 1100),
                                      (262144, 3), (262144, 18)])
def test_even_rows(n, length, hubs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf

    prdf.load()
    rng = np.random.default_rng(length + hubs)
    lens = np.full(n, length, np.int64)
    lens[rng.choice(n, hubs, replace=False)] = 7000
    if length > 2:  # every second row one shorter
        lens[::2] -= 1
    off = np.zeros(n + 1, np.int64)
    off[1:] = np.cumsum(lens)
    row = np.repeat(np.arange(n), lens)
    col = rng.integers(0, n, row.size)
    col[off[:-1]] = np.arange(n)  # a self-loop each, so that every vertex has an out-edge
    deg = np.bincount(col, minlength=n)
    iters = 4
    R = np.full(n, 1.0 / n)
    for _ in range(iters):
        new = 0.15 / n + 0.85 * np.bincount(row, (R / deg)[col], n)
        delta = np.abs(new - R).max()
        R = new
    p = prdf.pr_params_default()
    p.max_iter = iters
    p.tol = 0.0
    got = torch.empty(n, dtype=torch.float64, device="cuda")
    st = prdf.pr_static_noalloc(n, torch.from_numpy(off).cuda(), torch.from_numpy(col.astype(np.int32)).cuda(), got, p)
    assert st.iterations == iters or st.last_delta == 0.0  # (a fixed point)
    # a sum of k terms in any order is within k 2^-53 of itself, on either side; a division and three
    # more operations a row; errors of an iteration go on with a factor of at most 1
    eps = 2 * iters * (lens.max() + 4) * 2.0 ** -53 * R.max()
    assert np.abs(got.cpu().numpy() - R).max() <= eps
    assert abs(st.last_delta - delta) <= 2 * eps
