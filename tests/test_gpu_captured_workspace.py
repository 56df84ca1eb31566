"""A captured dash (with its list of round caps) and raster replay unharmed after larger calls on
the same context have outgrown every workspace that the graph was given."""
import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_replay_after_larger_calls():
    import torch
    import paper_2007_00308_gb300 as ps
    z = lambda shape, dt: torch.zeros(shape, dtype=dt, device="cuda")  # noqa: E731

    class Scene:
        def __init__(self, n_paths, room):
            b = W.c2_batching(n_paths=n_paths, canvas=512)
            self.db = ps.DeviceBatch(b)
            self.out = ps.tessellate(ps.Context(), self.db, ps.PS_PREC_MIXED, want_t=True)
            self.cap = room * self.out.capacity + 100000
            self.dash = [z((self.cap, 4), torch.float32), z(self.cap, torch.float32),
                         z(self.cap, torch.int32), z(self.cap, torch.int32), z(1, torch.int64)]
            self.canvas, self.covered = z((400, 512), torch.int16), z(n_paths, torch.int64)
            self.g_rib, self.g_s = torch.ones_like(self.out.rib), torch.ones_like(self.out.s)
            self.g_pts = z(self.db.n_seg * 8, torch.float32)
            self.g_w = z(n_paths, torch.float32)

        def calls(self, ctx, dtheta):
            o = self.out
            ps.ps_tessellate_strokes(ctx, self.db, o, ps.PS_PREC_MIXED)
            ps.ps_dash_capped(ctx, o.rib, o.s, o.tag, o.n_rib, o.capacity, [9.0, 3.0, 1.0, 3.0], 0.5,
                              self.db.path_cap, dtheta, *self.dash, self.cap)
            ps.ps_rasterize_coverage(ctx, self.dash[0], self.dash[2], self.dash[4], self.cap,
                                     self.db.n_path, 512, 400, self.canvas, self.covered)
            ps.ps_tessellate_backward(ctx, self.db, o, self.g_rib, self.g_s, self.g_pts, self.g_w,
                                      ps.PS_PREC_MIXED)

        def results(self):
            torch.cuda.synchronize()
            return [t.clone() for t in (*self.dash, self.out.rib, self.out.s, self.canvas, self.covered)]

    ctx = ps.Context()
    ctx.reserve(n_pair=8_000_000)
    small, large = Scene(20, 12), Scene(300, 12)
    small.calls(ctx, small.db.dtheta)
    assert ctx.status() == 0
    want = small.results()
    assert int(small.dash[4].item()) > 0
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        small.calls(ctx, small.db.dtheta)
    # larger in every way; coarser caps make for a longer list at the same output size
    ctx.reserve(n_pair=80_000_000)
    large.calls(ctx, 8 * large.db.dtheta)
    large.calls(ctx, 20 * large.db.dtheta)
    assert ctx.status() == 0
    # whatever has been given back is overwritten
    waste = [torch.full((n << 18,), -1, dtype=torch.int32, device="cuda")
             for n in (1, 4, 16, 64, 256) for _ in range(4)]
    for t in (*small.dash, small.canvas, small.covered, small.out.rib, small.out.s):
        t.zero_()
    g.replay()
    got = small.results()
    assert ctx.status() == 0
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert len(waste) == 20
