"""The calls' kernels overlap their launches: back-to-back calls without a wait, calls captured
into a graph and replayed, and calls with the profile's event records in between (which turn
the overlap off) all give the same ribs, dashes and coverage."""
import numpy as np
import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_paths", [1, 120])
def test_back_to_back_captured_and_profiled_agree(n_paths):
    import torch
    import paper_2007_00308_gb300 as ps
    batches = [W.c2_batching(n_paths=n_paths, seed=s, canvas=300) for s in (3, 4)]
    dbs = [ps.DeviceBatch(b) for b in batches]
    ctx = ps.Context()
    outs = [ps.tessellate(ctx, db, ps.PS_PREC_MIXED) for db in dbs]
    canvas = [torch.zeros((203, 300), dtype=torch.int16, device="cuda") for _ in dbs]
    covered = [torch.zeros(n_paths, dtype=torch.int64, device="cuda") for _ in dbs]
    cap = 4 * max(o.capacity for o in outs) + 4096
    dashed = [[torch.zeros((cap, 4), device="cuda"), torch.zeros(cap, device="cuda"),
               torch.zeros(cap, dtype=torch.int32, device="cuda"), None,
               torch.zeros(1, dtype=torch.int64, device="cuda")] for _ in dbs]
    ctx.reserve(n_pair=4_000_000)

    def calls():  # two different batches in turn on one context
        for db, o, cv, cd, d in zip(dbs, outs, canvas, covered, dashed):
            ps.ps_tessellate_strokes(ctx, db, o, ps.PS_PREC_MIXED)
            ps.ps_dash(ctx, o.rib, o.s, o.tag, o.n_rib, o.capacity, [5.0, 2.0], 0.0, *d, cap)
            ps.ps_rasterize_coverage(ctx, o.rib, o.tag, o.n_rib, o.capacity, n_paths, 300, 203, cv, cd)

    def state():
        torch.cuda.synchronize()
        assert ctx.status() == 0
        return [t.cpu().numpy().copy() for o, cv, cd, d in zip(outs, canvas, covered, dashed)
                for t in (o.rib, o.tag, o.s, o.path_len, cv, cd, d[0], d[1], d[2], d[4])]

    calls()
    want = state()
    assert any(w.any() for w in want)
    for _ in range(20):
        calls()
    got = state()
    ctx.profile(True)
    calls()
    profiled = state()
    ctx.profile(False)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        calls()
    for _ in range(3):
        g.replay()
    captured = state()
    for other in (got, profiled, captured):
        for a, r in zip(other, want):
            assert np.array_equal(a, r)
