"""A dash call captured first thing on a reserved context allocates nothing, writes its round
caps without the cap list, and gives what the eager call gives with it."""
import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("capped", [False, True])
def test_first_call_captured(capped):
    import torch
    import paper_2007_00308_gb300 as ps
    b = W.c2_batching(n_paths=60)
    ctx = ps.Context()
    db = ps.DeviceBatch(b)
    out = ps.tessellate(ctx, db, ps.PS_PREC_MIXED)
    cap = 12 * out.capacity + 200000

    def buffers():
        z = lambda shape, dt: torch.zeros(shape, dtype=dt, device="cuda")  # noqa: E731
        return [z((cap, 4), torch.float32), z(cap, torch.float32), z(cap, torch.int32),
                z(cap, torch.int32), z(1, torch.int64)]

    def dash(c, bufs):
        args = (*bufs, cap)
        if capped:
            ps.ps_dash_capped(c, out.rib, out.s, out.tag, out.n_rib, out.capacity, [9.0, 3.0, 1.0, 3.0],
                              0.5, db.path_cap, db.dtheta, *args)
        else:
            ps.ps_dash(c, out.rib, out.s, out.tag, out.n_rib, out.capacity, [9.0, 3.0, 1.0, 3.0], 0.5,
                       *args)

    want = buffers()
    dash(ctx, want)
    assert ctx.status() == 0
    fresh = ps.Context()
    fresh.reserve(n_link=db.n_link, n_rib=out.capacity)
    got = buffers()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        dash(fresh, got)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert fresh.status() == 0
    assert int(want[4].item()) > 0
    for a, r in zip(got, want):
        assert torch.equal(a, r)
