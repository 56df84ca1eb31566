"""tessellate() on another stream than the current one: its buffers are not written before the
current stream's earlier work is done with their memory, nor given back before its own is."""
import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu


class Bare:
    """A stream of another library: all that the calls ask for is its handle."""

    def __init__(self, stream):
        self.cuda_stream = stream.cuda_stream


@pytest.mark.parametrize("kind", ["stream", "bare", "current"])
def test_other_stream(kind):
    import torch
    import paper_2007_00308_gb300 as ps
    db = ps.DeviceBatch(W.c2_batching(n_paths=120))
    want = ps.tessellate(ps.Context(), db, ps.PS_PREC_MIXED)
    torch.cuda.synchronize()
    side = torch.cuda.current_stream() if kind == "current" else torch.cuda.Stream()
    stream = Bare(side) if kind == "bare" else side
    ctx = ps.Context()
    for _ in range(4):
        # blocks of every size, still being written on the current stream when they are given back
        waste = [torch.empty(1 << n, dtype=torch.uint8, device="cuda") for n in range(4, 27)]
        torch.cuda._sleep(10_000_000)
        for w in waste:
            w.fill_(255)
        del waste, w
        got = ps.tessellate(ctx, db, ps.PS_PREC_MIXED, stream=stream)
        over = [torch.full((1 << n,), 255, dtype=torch.uint8, device="cuda") for n in range(4, 27)]
        torch.cuda.synchronize()
        assert ctx.status() == 0 and len(over) == 23
        for name in ("rib", "tag", "s", "path_len", "link_rib_off", "path_rib_off", "n_rib"):
            assert torch.equal(getattr(got, name), getattr(want, name)), name
