"""A destroyed handle gives its device memory back, the device-side loops' too."""
import pytest

import __graft_entry__
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["static", "frontier", "frontier_async", "traversal"])
def test_destroyed_handles_leave_nothing(call):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    __graft_entry__.build()
    from paper_2401_03256_gb300 import prdf

    prdf.load()
    g = synth.rmat(13, 8, seed=1)
    b = synth.BatchStream(g, seed=2).next(5e-2)

    def one():
        with prdf.Graph(g.n, g.src, g.dst) as h:
            h.static()
            h.apply(b.del_src, b.del_dst, b.ins_src, b.ins_dst)
            getattr(h, call)()

    for _ in range(5):
        one()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(60):
        one()
    # a loop takes 0.9 MB; the driver hands memory out 2 MB at a time
    assert free - torch.cuda.mem_get_info()[0] <= 8 << 20
