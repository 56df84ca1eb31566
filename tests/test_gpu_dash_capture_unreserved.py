"""A dash captured on a context with no words for its quads brings its own."""
import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_first_call_captured_unreserved():
    """A context that has tessellated but never dashed, and reserved nothing: the graph brings
    its own words; instantiated, replayed and replayed again after the context has grown."""
    import torch
    import paper_2007_00308_gb300 as ps
    b = W.c2_batching(n_paths=8)
    ctx = ps.Context()
    db = ps.DeviceBatch(b)
    out = ps.tessellate(ctx, db, ps.PS_PREC_MIXED)
    cap = 3 * out.capacity + 20000

    def buffers():
        z = lambda shape, dt: torch.zeros(shape, dtype=dt, device="cuda")  # noqa: E731
        return [z((cap, 4), torch.float32), z(cap, torch.float32), z(cap, torch.int32),
                z(cap, torch.int32), z(1, torch.int64)]

    def dash(c, bufs):
        ps.ps_dash(c, out.rib, out.s, out.tag, out.n_rib, out.capacity, [9.0, 3.0, 1.0, 3.0], 0.5, *bufs, cap)

    want, got = buffers(), buffers()
    dash(ps.Context(), want)
    fresh = ps.Context()
    ps.ps_tessellate_strokes(fresh, db, out, ps.PS_PREC_MIXED)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        dash(fresh, got)
    for _ in range(2):
        for t in got:
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert fresh.status() == 0
        assert int(want[4].item()) > 0
        for a, r in zip(got, want):
            assert torch.equal(a, r)
        dash(fresh, buffers())
