"""Kernels launched while the one before still runs read what it wrote, and not what stood there:
calls on small and large batches in turn share every buffer, without a wait in between, and give
what each gives by itself in buffers of its own."""
import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PATTERN = [9.0, 3.0, 1.0, 3.0]


def test_shared_buffers_back_to_back():
    import torch
    import paper_2007_00308_gb300 as ps
    batches = [W.c2_batching(n_paths=n, seed=s, canvas=300) for s, n in enumerate((90, 1, 20, 200))]
    dbs = [ps.DeviceBatch(b) for b in batches]
    cap = max(ps.tessellate(ps.Context(), db, ps.PS_PREC_MIXED).capacity for db in dbs)
    dcap = 8 * cap + 200000

    class Buffers:
        def __init__(self):
            z = lambda shape, dt: torch.zeros(shape, dtype=dt, device="cuda")  # noqa: E731
            self.ctx = ps.Context()
            self.out = ps.TessOutput(max(d.n_link for d in dbs), max(d.n_path for d in dbs), cap,
                                     want_t=True)
            self.dash = [z((dcap, 4), torch.float32), z(dcap, torch.float32), z(dcap, torch.int32),
                         z(dcap, torch.int32), z(1, torch.int64)]
            self.canvas = z((203, 300), torch.int16)
            self.covered = z(max(d.n_path for d in dbs), torch.int64)

        def calls(self, db):
            o, d = self.out, self.dash
            ps.ps_tessellate_strokes(self.ctx, db, o, ps.PS_PREC_MIXED)
            ps.ps_dash_capped(self.ctx, o.rib, o.s, o.tag, o.n_rib, o.capacity, PATTERN, 0.0,
                              db.path_cap, db.dtheta, *d, dcap)
            ps.ps_rasterize_coverage(self.ctx, d[0], d[2], d[4], dcap, db.n_path, 300, 203, self.canvas,
                                     self.covered)

        def results(self, db):
            o, d = self.out, self.dash
            n, m = o.n_rib.clone(), d[4].clone()
            return n, m, [o.rib.clone(), o.tag.clone(), o.s.clone(), o.t.clone(), o.path_len.clone(),
                          d[0].clone(), d[1].clone(), d[2].clone(), d[3].clone(), self.canvas.clone(),
                          self.covered.clone()]

    want = []
    for db in dbs:
        own = Buffers()
        own.ctx.reserve(n_pair=80_000_000)
        own.calls(db)
        torch.cuda.synchronize()
        assert own.ctx.status() == 0
        want.append(own.results(db))
    shared = Buffers()
    shared.ctx.reserve(n_pair=80_000_000)
    torch.cuda.synchronize()
    got = []
    for _ in range(3):
        for db in dbs:
            shared.calls(db)
            got.append(shared.results(db))
    torch.cuda.synchronize()
    assert shared.ctx.status() == 0
    for i, (n, m, parts) in enumerate(got):
        db, (n0, m0, parts0) = dbs[i % len(dbs)], want[i % len(dbs)]
        assert n.item() == n0.item() > 0 and m.item() == m0.item() > 0
        rows = [n.item()] * 4 + [db.n_path] + [m.item()] * 4 + [203, db.n_path]
        for k, a, b in zip(rows, parts, parts0):
            assert torch.equal(a[:k], b[:k])
