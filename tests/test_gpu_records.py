"""The tessellation over the links' records (one set-up for count, ribs and adjoint) against
the calls that set the links up themselves, and PolarStroke's upstream gradients in
the forms that reach it: dense, expanded, transposed, off a 16-byte boundary, absent."""
import numpy as np
import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _batches():
    yield W.c2_batching(n_paths=40)
    yield W.c5_differentiation(n_paths=7, n_seg=5)
    yield W.single([W.LINE], [[[3, 3], [3, 3], [3, 3], [3, 3]]])  # one zero-length segment: no ribs


@pytest.mark.parametrize("tau", [0.0, 0.25])
@pytest.mark.parametrize("precision", [0, 1])
def test_ribs_from_records_are_the_tessellation(precision, tau):
    import torch
    import paper_2007_00308_gb300 as ps
    for b in _batches():
        ctx = ps.Context()
        ctx.set_pixel_tolerance(tau)
        db = ps.DeviceBatch(b)
        got = ps.tessellate(ctx, db, precision, want_t=True)
        ref = ps.TessOutput(db.n_link, db.n_path, got.capacity, want_t=True)
        ps.ps_tessellate_strokes(ctx, db, ref, precision)
        assert ctx.status() == 0
        R = int(ref.n_rib.item())
        assert R == int(got.n_rib.item()) and got.capacity == max(R, 1)
        for name in ("rib", "tag", "s", "t"):
            assert torch.equal(getattr(got, name)[:R], getattr(ref, name)[:R]), name
        for name in ("link_rib_off", "path_rib_off", "path_len"):
            assert torch.equal(getattr(got, name), getattr(ref, name)), name


def _reference_grads(ps, torch, b, g_rib, g_s):
    ctx, db = ps.Context(), ps.DeviceBatch(b)
    out = ps.tessellate(ctx, db, ps.PS_PREC_MIXED, want_t=True)
    gp = torch.empty(db.n_seg * 8, device="cuda")
    gw = torch.empty(db.n_path, device="cuda")
    ps.ps_tessellate_backward(ctx, db, out, g_rib.contiguous().clone(), g_s.contiguous().clone(), gp, gw)
    return gp.cpu().numpy(), gw.cpu().numpy()


@pytest.mark.parametrize("form", ["dense", "expanded", "transposed", "unaligned", "rib only", "s only"])
def test_upstream_gradients_in_every_form(form):
    import torch
    import paper_2007_00308_gb300 as ps
    from paper_2007_00308_gb300.autograd import PolarStroke
    b = W.c5_differentiation(n_paths=5, n_seg=4)
    pts = torch.from_numpy(b.seg_pts).cuda().requires_grad_(True)
    width = torch.from_numpy(b.path_width).cuda().requires_grad_(True)
    rib, s = PolarStroke.apply(pts, width, b)
    R = rib.shape[0]
    gen = torch.Generator(device="cuda").manual_seed(3)
    g_rib = torch.randn((R, 4), generator=gen, device="cuda")
    g_s = torch.randn(R, generator=gen, device="cuda")
    outs, ups = (rib, s), (g_rib, g_s)
    if form == "expanded":
        ups = (torch.ones((), device="cuda").expand(R, 4), torch.ones((), device="cuda").expand(R))
    elif form == "transposed":
        ups = (g_rib.t().contiguous().t(), g_s)
    elif form == "unaligned":
        ups = (torch.cat([g_rib.new_zeros(1), g_rib.reshape(-1)])[1:].view(R, 4),
               torch.cat([g_s.new_zeros(1), g_s])[1:])
        assert ups[0].data_ptr() % 16 and ups[1].data_ptr() % 16
    elif form == "rib only":
        outs, ups = (rib,), (g_rib,)
    elif form == "s only":
        outs, ups = (s,), (g_s,)
    got = torch.autograd.grad(outs, (pts, width), ups)
    full = (ups[0] if form != "s only" else torch.zeros_like(g_rib),
            ups[-1] if form != "rib only" else torch.zeros_like(g_s))
    ref = _reference_grads(ps, torch, b, *full)
    for a, r in zip(got, ref):
        a = a.cpu().numpy().reshape(-1)
        # the two differ by the order of the FP32 atomic sums
        assert np.abs(a - r).max() <= 1e-5 * max(np.abs(r).max(), 1e-6)


def test_no_ribs_no_gradient():
    import torch
    from paper_2007_00308_gb300.autograd import PolarStroke
    b = W.single([W.LINE], [[[3, 3], [3, 3], [3, 3], [3, 3]]])
    pts = torch.from_numpy(b.seg_pts).cuda().requires_grad_(True)
    width = torch.from_numpy(b.path_width).cuda().requires_grad_(True)
    rib, s = PolarStroke.apply(pts, width, b)
    assert rib.shape == (0, 4) and s.shape == (0,)
    g = torch.autograd.grad((rib.sum() + s.sum()), (pts, width))
    assert not g[0].any() and not g[1].any()
