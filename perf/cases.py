"""The calls whose speed counts: what programs have the stroking library do.

A case is a dict of plain values.  ``kind`` says which calls a pass makes:

* ``picture``     tessellate a batch of paths and rasterize the strokes (16 samples per pixel)
* ``dashes``      tessellate, dash by arc length (butt or capped dash ends), optionally rasterize
* ``tessellate``  ribs, tags and arc length alone (a renderer or a cutter takes them from there)
* ``fit``         ribs and arc length as differentiable tensors, and their gradients

``shape`` says what is stroked: ``mixed`` (random walks of lines, quadratics, cubics and conics
with exact cusps and loops, widths of 0.5 to 64 px, several joins and caps), ``curves`` (chained
random cubics), ``walk`` (one long random walk of cubics), ``near_cusp`` (single cubics next to
cusps and collinearity, far from the origin).  Sizes are those of the seeded workloads of
``paper_2007_00308_gb300/workloads.py``, of the tests and of the README, or lie between them.
"""
import math

import numpy as np
import torch

import paper_2007_00308_gb300 as ps
from paper_2007_00308_gb300 import autotune
from paper_2007_00308_gb300 import workloads as W

_LOOP = np.array([[0.0, 0.0], [1.5, 1.0], [-0.5, 1.0], [1.0, 0.0]])
_CUSP = np.array([[0.0, 0.0], [1.0, 1.0], [0.0, 1.0], [1.0, 0.0]])
_DASHES = {"dash": [12.0, 6.0], "dash_dot": [9.0, 3.0, 1.0, 3.0]}


def _case(kind, shape, paths, segments, step_deg, width=0, height=0, precision="mixed",
          stroke=8.0, closed=False, exact_quads=False, pixel_tol=0.0, dash="", capped=False,
          **more):
    return dict(kind=kind, shape=shape, paths=paths, segments=segments, step_deg=step_deg,
                width=width, height=height, precision=precision, stroke=stroke, closed=closed,
                exact_quads=exact_quads, pixel_tol=pixel_tol, dash=dash, capped=capped, **more)


def listed():
    return [
        # one curve on a small canvas: an interactive editor's redraw, all latency
        _case("picture", "curves", 1, 1, 2.0, 256, 256, stroke=12.0, name="one curve"),
        # an icon or a glyph run: one path of 64 chained cubics
        _case("picture", "curves", 1, 64, 2.0, 512, 512, name="icon"),
        # an ordinary drawing of a few hundred paths on an odd-sized window
        _case("picture", "mixed", 300, 30, 1.0, 1003, 747, name="drawing"),
        # the library's benchmark: a map or a CAD sheet of 10,000 paths
        _case("picture", "mixed", 10000, 30, 1.0, 2048, 2048, name="dense sheet"),
        # quads filled by the crossing rule (bow-ties as such), full-HD: 1080 is no multiple of 16
        _case("picture", "mixed", 1000, 30, 1.0, 1920, 1080, exact_quads=True, name="crossing rule"),
        # a viewer's preview: the step grows towards pixel scale
        _case("picture", "mixed", 3000, 30, 1.0, 1601, 1199, pixel_tol=0.25, name="preview"),
        # one long path, thin and dashed, on a large canvas: a plotter or a route on a map
        _case("dashes", "walk", 1, 5031, 0.5, 4096, 4096, stroke=2.0, dash="dash", name="long dashed path"),
        # many short dashed paths with capped dash ends, handed on without a raster
        _case("dashes", "mixed", 1000, 30, 1.0, 2048, 2048, dash="dash_dot", capped=True, name="capped dashes"),
        # a million cubics next to cusps and flatness, coordinates up to 10^6
        _case("tessellate", "near_cusp", 1000000, 1, 1.0, stroke=1.0, name="near cusps"),
        # all-FP32 ribs for a preview that needs no more
        _case("tessellate", "curves", 2048, 32, 2.0, 1024, 1024, precision="fp32", name="single precision"),
        # a step of fitting a few strokes to a drawing: forward and gradients
        _case("fit", "curves", 16, 32, 2.0, 1024, 1024, name="small fit"),
        # the same for thousands of strokes at once
        _case("fit", "curves", 4096, 32, 2.0, 1024, 1024, name="large fit"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    step = rng.choice([0.5, 1.0, 2.0, 4.0])
    precision = "fp32" if rng.random() < 0.15 else "mixed"
    kind = rng.choice(["picture", "picture", "picture", "dashes", "tessellate", "fit"])
    w, h = log(200, 2048), log(200, 2048)
    if kind == "picture":
        more = dict(precision=precision, exact_quads=rng.random() < 0.25,
                    pixel_tol=rng.choice([0.0, 0.0, 0.0, 0.1, 0.25]))
        if rng.random() < 0.35:  # icons and glyph runs
            return _case(kind, "curves", log(1, 30), log(1, 64), step, w, h,
                         stroke=rng.choice([1.5, 4.0, 8.0, 12.0]), closed=rng.random() < 0.4, **more)
        # the sheet's paths per area, or fewer
        most = max(20.0, 8000.0 * w * h / 2048 ** 2)
        return _case(kind, "mixed", log(10, most), 30, max(step, 1.0), w, h, **more)
    if kind == "dashes":
        dash = rng.choice(sorted(_DASHES))
        if rng.random() < 0.5:
            return _case(kind, "walk", 1, log(50, 8000), step, 4 * (w // 2), 4 * (h // 2), stroke=2.0,
                         dash=dash, capped=rng.random() < 0.3)
        return _case(kind, "mixed", log(10, 2000), 30, max(step, 1.0), w, h, dash=dash,
                     capped=rng.random() < 0.5)
    if kind == "tessellate":
        shape = rng.choice(["mixed", "curves", "near_cusp"])
        n = log(100, 300000)
        if shape == "near_cusp":
            return _case(kind, shape, n, 1, max(step, 1.0), stroke=1.0, precision=precision)
        return _case(kind, shape, max(1, n // 32), 30 if shape == "mixed" else 32, max(step, 1.0),
                     1024, 1024, precision=precision)
    return _case(kind, "curves", log(4, 4000), log(4, 32), max(step, 1.0), 1024, 1024)


# ---- what is stroked ----------------------------------------------------------------
def _unit(a):
    return np.stack([np.cos(a), np.sin(a)], -1)


def _grid(v):
    return np.round(v * 64.0) / 64.0


def _walk(rng, counts, box, first_lo=0.0, first_hi=1.0):
    """Random walks of all paths at once: per segment start, end, step length and the headings
    before and after it; steps log-uniform 1 to 200 px, bounced off the canvas edges."""
    P, n_max = len(counts), int(counts.max())
    a = _grid(rng.uniform(first_lo, first_hi, (P, 2)) * box)
    h = rng.uniform(-math.pi, math.pi, P)
    rows = []
    for _ in range(n_max):
        L = np.exp(rng.uniform(0.0, math.log(200.0), P))
        before = h
        h = h + rng.uniform(-math.pi, math.pi, P)
        d = a + L[:, None] * _unit(h)
        h = np.where((d[:, 0] < 0) | (d[:, 0] > box[0]), math.pi - h, h)
        h = np.where((d[:, 1] < 0) | (d[:, 1] > box[1]), -h, h)
        d = _grid(np.clip(a + L[:, None] * _unit(h), 0.0, box))
        rows.append(np.concatenate([a, d, L[:, None], before[:, None], h[:, None]], 1))
        a = d
    inside = np.arange(n_max)[None, :] < counts[:, None]
    rows = np.stack(rows, 1)[inside]
    return rows[:, 0:2], rows[:, 2:4], rows[:, 4], rows[:, 5], rows[:, 6]


def _counts(case):
    """Segments per path, geometric with at most 200: the distribution's quantiles, so that a
    case has as many segments whatever the seed."""
    if case["shape"] != "mixed":
        return np.full(case["paths"], case["segments"])
    at = (np.arange(case["paths"]) + 0.5) / case["paths"]
    return np.clip(np.ceil(np.log1p(-at) / math.log1p(-1.0 / case["segments"])), 1, 200).astype(int)


def _mixed(case, rng):
    P, box = case["paths"], np.array([case["width"], case["height"]], float)
    counts = rng.permutation(_counts(case))
    a, d, L, before, after = _walk(rng, counts, box)
    S = len(L)
    kind = rng.choice([W.LINE, W.QUAD, W.CUBIC, W.CONIC], size=S, p=[0.2, 0.2, 0.45, 0.15])
    weight = np.where(kind == W.CONIC, np.exp(rng.uniform(math.log(0.1), math.log(10.0), S)), 1.0)
    half = math.pi / 2
    pts = np.stack([a, a, d, d], 1)  # lines
    mid = _grid(a + (L / 2)[:, None] * _unit(before + rng.uniform(-half, half, S)))
    third = (L / 3)[:, None]
    b = _grid(a + third * _unit(before + rng.uniform(-half, half, S)))
    c = _grid(d - third * _unit(after + rng.uniform(-half, half, S)))
    e = d - a
    q = _LOOP[None] * np.stack([np.ones(S), rng.choice([-1.0, 1.0], S)], 1)[:, None]
    loop = _grid(a[:, None] + np.stack([q[..., 0] * e[:, None, 0] - q[..., 1] * e[:, None, 1],
                                        q[..., 0] * e[:, None, 1] + q[..., 1] * e[:, None, 0]], -1))
    special = rng.uniform(0, 1, S) + np.where((e == 0).all(1), 1.0, 0.0)
    conic = (kind == W.QUAD) | (kind == W.CONIC)
    pts[conic, 1] = pts[conic, 2] = mid[conic]
    cubic = kind == W.CUBIC
    pts[cubic, 1], pts[cubic, 2] = b[cubic], c[cubic]
    cusp = cubic & (special < 0.1)  # C = A + B - D: g'(1/2) = 0
    b2 = np.where((b == d).all(1)[:, None], b + 1.0 / 64, b)
    pts[cusp, 1], pts[cusp, 2] = b2[cusp], (a + b2 - d)[cusp]
    loops = cubic & (special >= 0.1) & (special < 0.2)
    pts[loops, 1], pts[loops, 2] = loop[loops, 1], loop[loops, 2]
    return W.make_batch("mixed", kind, pts, weight, counts,
                        np.exp(rng.uniform(math.log(0.5), math.log(64.0), P)),
                        rng.choice([W.JOIN_MITER, W.JOIN_ROUND, W.JOIN_BEVEL], P),
                        rng.choice([W.CAP_BUTT, W.CAP_SQUARE, W.CAP_ROUND], P), 4.0, 0,
                        case["step_deg"])


def _curves(case, rng):
    P, n = case["paths"], case["segments"]
    box = np.array([case["width"], case["height"]], float)
    pts = (rng.random((P, n, 4, 2), dtype=np.float32) * box).astype(np.float32)
    pts[:, 1:, 0] = pts[:, :-1, 3]
    if case["closed"]:
        pts[:, -1, 3] = pts[:, 0, 0]
    widths = rng.uniform(1, 16, P) if P > 1 else case["stroke"]
    return W.make_batch("curves", np.full(P * n, W.CUBIC), pts, np.ones(P * n), np.full(P, n), widths,
                        W.JOIN_ROUND, W.CAP_ROUND, closed=int(case["closed"]),
                        dtheta_deg=case["step_deg"])


def _long_walk(case, rng):
    n, box = case["segments"], np.array([case["width"], case["height"]], float)
    a, d, L, before, after = _walk(rng, np.array([n]), box, 0.25, 0.75)
    half = math.pi / 2
    b = a + (L / 3)[:, None] * _unit(before + rng.uniform(-half, half, n))
    c = d - (L / 3)[:, None] * _unit(after + rng.uniform(-half, half, n))
    return W.make_batch("walk", np.full(n, W.CUBIC), np.stack([a, b, c, d], 1), np.ones(n), [n],
                        case["stroke"], W.JOIN_ROUND, W.CAP_ROUND, dtheta_deg=case["step_deg"])


def _near_cusp(case, rng):
    n = case["paths"]
    scale = np.exp(rng.uniform(math.log(0.1), math.log(1e3), n))
    rot = rng.uniform(-math.pi, math.pi, n)
    unit = np.zeros((n, 4, 2))
    unit[: n // 2] = _CUSP
    unit[n // 2:, 1:3, 0] = rng.uniform(-0.5, 1.5, (n - n // 2, 2))
    unit[n // 2:, 3, 0] = 1.0
    cs, sn = np.cos(rot)[:, None], np.sin(rot)[:, None]
    pts = np.stack([unit[..., 0] * cs - unit[..., 1] * sn, unit[..., 0] * sn + unit[..., 1] * cs], -1)
    moved = np.exp(rng.uniform(math.log(1e-6), math.log(1e-2), (n, 4, 2)))
    pts = (pts + moved * rng.choice([-1.0, 1.0], (n, 4, 2))) * scale[:, None, None]
    pts += rng.uniform(-1e6, 1e6, (n, 1, 2))
    return W.make_batch("near_cusp", np.full(n, W.CUBIC), pts, np.ones(n), np.ones(n, np.int64),
                        case["stroke"], W.JOIN_ROUND, W.CAP_BUTT, dtheta_deg=case["step_deg"])


_SHAPES = {"mixed": _mixed, "curves": _curves, "walk": _long_walk, "near_cusp": _near_cusp}


def _batch(case, seed):
    return _SHAPES[case["shape"]](case, np.random.Generator(np.random.PCG64(seed)))


#: Degrees that one segment turns on average, its join and its share of the caps included.
_TURN = {"mixed": 145.0, "curves": 310.0, "walk": 210.0, "near_cusp": 205.0}


def _room(case):
    """Room for a case's ribs whatever the seed: the static bound of a small batch, the average
    and a margin for a large one."""
    segs = int(_counts(case).sum())
    if segs < 3000:
        return ps.ps_max_ribs(segs, case["paths"], W.f32(math.radians(case["step_deg"])))
    return int(1.25 * segs * (_TURN[case["shape"]] / case["step_deg"] + 6))


def _dash_room(case):
    """The same for the dashed ribs: two per quad, the pieces cut off at stretch ends, and caps
    there (round ones on a third of the paths, when there are many); a segment of about 50 px
    has six stretches or fewer."""
    stretches = 50 * case["paths"] + 8 * int(_counts(case).sum())
    cap = int(180.0 / case["step_deg"]) + 6
    ends = 4 if not case["capped"] else cap if case["paths"] > 200 else 2 * cap
    return 2 * _room(case) + stretches * ends


def _upstream(case, seed):
    """Gradients of a loss with respect to the ribs and the arc length."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    n = _room(case)
    return (torch.randn((n, 4), generator=gen, device="cuda") * 0.01,
            torch.randn(n, generator=gen, device="cuda") * 0.001)


# ---- the passes ----------------------------------------------------------------------
def prepare(case, seed):
    """Inputs on the GPU, a context with its workspace, and output buffers with room for any
    batch of the case, as a program that strokes every frame keeps them."""
    batch = _batch(case, seed)
    ctx = ps.Context()
    ctx.set_pixel_tolerance(case["pixel_tol"])
    prec = ps.PS_PREC_FP32 if case["precision"] == "fp32" else ps.PS_PREC_MIXED
    st = dict(case=case, ctx=ctx, precision=prec)
    if case["kind"] == "fit":
        from paper_2007_00308_gb300.autograd import PolarStroke
        pts = torch.from_numpy(batch.seg_pts).cuda().requires_grad_(True)
        width = torch.from_numpy(batch.path_width).cuda().requires_grad_(True)
        return dict(st, stroke=PolarStroke.apply, batch=batch, pts=pts, width=width,
                    upstream=_upstream(case, seed))
    db = st["db"] = ps.DeviceBatch(batch)
    out = st["out"] = ps.TessOutput(db.n_link, db.n_path, _room(case))
    for unused in (out.rib, out.tag, out.s):  # what lies past the last rib
        unused.zero_()
    if case["kind"] == "dashes":
        st["pattern"] = _DASHES[case["dash"]]
        st["dashed"] = _dash_buffers(_dash_room(case))
    if _rasterizes(case):
        w, h = case["width"], case["height"]
        st["canvas"] = torch.zeros((h, w), dtype=torch.int16, device="cuda")
        st["covered"] = torch.zeros(db.n_path, dtype=torch.int64, device="cuda")
        run(st)
        pairs = ps.ps_raster_stats(ctx)["pairs"]
        ctx.status()  # a first pass may have had too few bins
        autotune.reserve_bins(ctx, ((w + 15) // 16) * ((h + 15) // 16), pairs)
    run(st)
    status = ctx.status()
    if status:
        raise RuntimeError(f"prepare: {ps.error_string(status)}")
    return st


def _rasterizes(case):
    return case["kind"] == "picture" or (case["kind"] == "dashes" and not case["capped"])


def _dash_buffers(capacity):
    new = lambda shape, dtype: torch.zeros(shape, dtype=dtype, device="cuda")  # noqa: E731
    return dict(rib=new((capacity, 4), torch.float32), s=new(capacity, torch.float32),
                tag=new(capacity, torch.int32), src=new(capacity, torch.int32),
                n=new(1, torch.int64))


def _dash(st):
    o, d = st["out"], st["dashed"]
    args = (d["rib"], d["s"], d["tag"], d["src"], d["n"], d["rib"].shape[0])
    if st["case"]["capped"]:
        ps.ps_dash_capped(st["ctx"], o.rib, o.s, o.tag, o.n_rib, o.capacity, st["pattern"], 0.0,
                          st["db"].path_cap, st["db"].dtheta, *args)
    else:
        ps.ps_dash(st["ctx"], o.rib, o.s, o.tag, o.n_rib, o.capacity, st["pattern"], 0.0, *args)


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "fit":
        rib, s = state["stroke"](state["pts"], state["width"], state["batch"], state["precision"], ctx)
        g_rib, g_s = state["upstream"]
        n = rib.shape[0]
        g = torch.autograd.grad((rib, s), (state["pts"], state["width"]), (g_rib[:n], g_s[:n]))
        return dict(grad_pts=g[0], grad_width=g[1])
    db, out = state["db"], state["out"]
    ps.ps_tessellate_strokes(ctx, db, out, state["precision"])
    got = dict(rib=out.rib, tag=out.tag, s=out.s, link_rib_off=out.link_rib_off,
               path_rib_off=out.path_rib_off, path_len=out.path_len, n_rib=out.n_rib)
    rib, tag, n, capacity = out.rib, out.tag, out.n_rib, out.capacity
    if case["kind"] == "dashes":
        _dash(state)
        d = state["dashed"]
        rib, tag, n, capacity = d["rib"], d["tag"], d["n"], d["rib"].shape[0]
        got["dashed"] = d
    if "canvas" in state:
        ps.ps_rasterize_coverage(ctx, rib, tag, n, capacity, db.n_path, case["width"], case["height"],
                                 state["canvas"], state["covered"], exact=case["exact_quads"])
        got.update(canvas=state["canvas"], covered=state["covered"])
    return got


def work(case):
    """What a pass cannot do without: the inputs read and the outputs written once, and per rib
    its angle, its t and its two vertices in single precision."""
    segs = int(_counts(case).sum())
    ribs = segs * (_TURN[case["shape"]] / case["step_deg"] + 3) * (0.6 if case["pixel_tol"] else 1.0)
    moved = 37 * segs + 18 * case["paths"] + 24 * ribs + 8 * segs
    flops = 100 * ribs
    if case["kind"] == "fit":  # upstream gradients in, gradients out
        moved += 20 * ribs + 32 * segs + 4 * case["paths"]
        flops += 150 * ribs
    if case["kind"] == "dashes":  # about two thirds of the quads, two ribs each
        moved += 28 * 1.3 * ribs
        flops += 30 * ribs
    if _rasterizes(case):
        moved += 2 * case["width"] * case["height"] + 8 * case["paths"]
        flops += 16 * 4 * ribs  # a quad of about a pixel, four edges each
    return {"bytes": moved, "flops": flops}


# ---- 64-bit values ----------------------------------------------------------------------
def exact(case, seed):
    """Ribs, arc length and gradients in 64 bits, for open paths of cubics in general position
    with round joins and caps (shapes "curves" and "walk"); the rest has None, and so have
    all-FP32 ribs, whose step counts are decided in single precision."""
    if case["shape"] not in ("curves", "walk") or case["closed"] or case["pixel_tol"]:
        return None
    if case["precision"] == "fp32":
        return None
    if case["paths"] * case["segments"] > 150000:
        return None
    batch = _batch(case, seed)
    q, off = batch.dtheta, batch.path_seg_off.astype(np.int64)
    fit = case["kind"] == "fit"
    at = list(range(0, batch.n_path, 512)) + [batch.n_path]
    parts = []
    for p0, p1 in zip(at, at[1:]):
        pts = torch.from_numpy(batch.seg_pts[off[p0]:off[p1]]).cuda().double().requires_grad_(fit)
        width = torch.from_numpy(batch.path_width[p0:p1]).cuda().double().requires_grad_(fit)
        n = torch.from_numpy(np.diff(off[p0:p1 + 1])).cuda()
        with torch.set_grad_enabled(fit):
            parts.append((pts, width) + _stroke64(pts, width, n, q))
    if fit:
        g_rib, g_s = _upstream(case, seed)
        grads, k = [], 0
        for p in parts:
            e = k + p[2].shape[0]
            grads.append(torch.autograd.grad(
                (p[2], p[3]), (p[0], p[1]), (g_rib[k:e].double(), g_s[k:e].double())))
            k = e
        return dict(grad_pts=torch.cat([g[0] for g in grads]),
                    grad_width=torch.cat([g[1] for g in grads]))
    rib, s = torch.cat([p[2] for p in parts]), torch.cat([p[3] for p in parts])
    unused = _room(case) - rib.shape[0]
    rib, s = torch.nn.functional.pad(rib, (0, 0, 0, unused)), torch.nn.functional.pad(s, (0, unused))
    got = dict(rib=rib, tag=None, s=s, link_rib_off=None, path_rib_off=None,
               path_len=torch.cat([p[4] for p in parts]), n_rib=None)
    if case["kind"] == "dashes":
        got["dashed"] = None
    if case["kind"] == "picture":
        got.update(canvas=None, covered=None)
    return got


def _cross(a, b):
    return a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]


def _angle(v):
    return torch.atan2(v[..., 1], v[..., 0])


def _roots(a, b, c):
    """Real roots of a + b t + c t^2, NaN where there are none."""
    disc = b * b - 4 * a * c
    real = disc > 0
    sq = torch.where(real, disc, torch.ones_like(disc)).sqrt()
    m = -0.5 * (b + torch.where(b >= 0, sq, -sq))
    nan = torch.full_like(a, math.nan)
    return torch.where(real, m / c, nan), torch.where(real, a / m, nan)


def _tangent(e, t):
    """g'(t) / 3 of a cubic with the control polygon's legs e [..., 3, 2]."""
    t = t[..., None]
    u = 1 - t
    return e[..., 0, :] * u * u + e[..., 1, :] * (2 * u * t) + e[..., 2, :] * t * t


def _solve(e, psi, lo, hi):
    """t in [lo, hi] where the tangent points along psi."""
    sn, cs = torch.sin(psi), torch.cos(psi)
    h = e[..., 1] * cs[..., None] - e[..., 0] * sn[..., None]  # legs against the normal
    r = torch.stack(_roots(h[..., 0], 2 * (h[..., 1] - h[..., 0]), h[..., 0] - 2 * h[..., 1] + h[..., 2]), -1)
    with torch.no_grad():
        ok = (r >= lo[..., None] - 1e-9) & (r <= hi[..., None] + 1e-9)
        H = _tangent(e[..., None, :, :], torch.nan_to_num(r))
        along = torch.where(ok, H[..., 0] * cs[..., None] + H[..., 1] * sn[..., None], -math.inf)
        best = along.argmax(-1, keepdim=True)
        ends = [(_cross(_tangent(e, t), torch.stack([cs, sn], -1))).abs() for t in (lo, hi)]
        some = ok.any(-1)
    return torch.where(some, r.gather(-1, best)[..., 0], torch.where(ends[0] < ends[1], lo, hi))


def _steps(turn, q):
    return torch.ceil(turn.detach().abs() / q - 1e-4).long().clamp(min=1)


def _stroke64(pts, width, n_seg, q):
    """Polar stroking of open cubic paths, round joins and caps: ribs, arc length, path lengths."""
    S, P, dev = pts.shape[0], n_seg.shape[0], pts.device
    path = torch.repeat_interleave(torch.arange(P, device=dev), n_seg)
    first = torch.cumsum(n_seg, 0) - n_seg
    e = pts[:, 1:] - pts[:, :-1]
    # intervals between inflections, their turnings, split where a half turn is reached
    l1, l2, l3 = _cross(e[:, 0], e[:, 1]), _cross(e[:, 0], e[:, 2]), _cross(e[:, 1], e[:, 2])
    a, b, c = l1, l2 - 2 * l1, l1 - l2 + l3
    r = torch.stack(_roots(a, b, c), -1)
    r = torch.where((r > 0) & (r < 1), r, torch.ones_like(r))  # none: an empty interval at 1
    r = torch.gather(r, 1, torch.argsort(r.detach(), 1))
    one = torch.ones_like(l1)
    p = torch.stack([0 * one, r[:, 0], r[:, 1], one], 1)
    end = _angle(e[:, 2])
    Psi = torch.stack([_angle(e[:, 0])] + [torch.where(p[:, k] < 1, _angle(_tangent(e, p[:, k])), end)
                                           for k in (1, 2)] + [end], 1)
    mid = 0.5 * (p[:, 1:] + p[:, :-1])
    sign = torch.sign(a[:, None] + b[:, None] * mid + c[:, None] * mid * mid).detach()
    d = sign * (Psi[:, 1:] - Psi[:, :-1])
    turn = sign * (d - 2 * math.pi * torch.floor(d.detach() / (2 * math.pi)))
    there = (p[:, 1:] > p[:, :-1]).detach()
    split = (turn.abs() >= math.pi).detach() & there
    part = torch.where(split, 0.5 * turn, turn)
    psi_s = Psi[:, :-1] + part
    t_s = torch.where(split, _solve(e[:, None].expand(-1, 3, -1, -1), psi_s, p[:, :-1], p[:, 1:]), p[:, 1:])
    count = torch.where(there, _steps(part, q), 0)
    count = torch.stack([count, torch.where(split, count, 0)], 2).reshape(S, 6)
    p0 = torch.cat([torch.stack([p[:, :-1], t_s], 2).reshape(S, 6), one[:, None]], 1)
    psi0 = torch.cat([torch.stack([Psi[:, :-1], psi_s], 2).reshape(S, 6), end[:, None]], 1)
    hi = torch.stack([t_s, p[:, 1:]], 2).reshape(S, 6)
    step = torch.repeat_interleave(part, 2, 1) / count.clamp(min=1)
    cum = torch.cat([torch.zeros((S, 1), dtype=torch.long, device=dev), torch.cumsum(count, 1)], 1)
    # joins (after every segment but a path's last) and caps
    last = first + n_seg - 1
    is_last = torch.zeros(S, dtype=torch.bool, device=dev)
    is_last[last] = True
    nxt = torch.where(is_last, torch.arange(S, device=dev), torch.arange(S, device=dev) + 1)
    bend = torch.atan2(_cross(e[:, 2], e[nxt, 0]), (e[:, 2] * e[nxt, 0]).sum(-1))
    cap = int(math.ceil(math.pi / q - 1e-4))
    # links in order: start cap, segment, join, ..., segment, end cap
    seg_link = 2 * torch.arange(S, device=dev) + path + 1
    start_link, end_link = seg_link[first] - 1, seg_link[last] + 1
    ribs = torch.full((2 * S + P,), cap + 1, dtype=torch.long, device=dev)
    ribs[seg_link] = cum[:, 6] + 1
    inner = torch.nonzero(~is_last)[:, 0]
    ribs[seg_link[inner] + 1] = _steps(bend[inner], q) + 1
    off = torch.cumsum(ribs, 0) - ribs
    R = int(ribs.sum())

    def spread(links):  # rib indexes of the links, the link of each (as an index into links), j
        which = torch.repeat_interleave(torch.arange(len(links), device=dev), ribs[links])
        k = torch.arange(len(which), device=dev)
        j = k - (torch.cumsum(ribs[links], 0) - ribs[links])[which]
        return off[links][which] + j, which, j

    def both(at, psi, rn, rp):
        n = torch.stack([-torch.sin(psi), torch.cos(psi)], -1)
        return torch.cat([at - rn[:, None] * n, at + rp[:, None] * n], 1)

    idx, s, j = spread(seg_link)
    k = (cum[s, 1:] <= j[:, None]).sum(1)
    m = k.clamp(max=5)
    since = (j - cum[s, k]).double()
    psi = psi0[s, k] + torch.where(since > 0, step[s, m] * since, 0.0)
    t = torch.where(since > 0, _solve(e[s], psi, p0[s, m], hi[s, m]), p0[s, k])
    u, tt = (1 - t)[:, None], t[:, None]
    rel = 3 * u * u * tt * (pts[s, 1] - pts[s, 0]) + 3 * u * tt * tt * (pts[s, 2] - pts[s, 0]) \
        + tt ** 3 * (pts[s, 3] - pts[s, 0])
    r = 0.5 * width[path[s]]
    rib = torch.zeros((R, 4), dtype=torch.float64, device=dev)
    rib = rib.index_put((idx,), both(pts[s, 0] + rel, psi, r, r))
    move = rel[1:] - rel[:-1]
    sq = (move * move).sum(-1)
    go = ((j[1:] > 0) & (t[1:] >= t[:-1]) & (sq > 0)).detach()
    chord = torch.where(go, torch.where(go, sq, 1.0).sqrt(), 0.0)
    length = torch.cumsum(torch.zeros(R, dtype=torch.float64, device=dev).index_put((idx[1:],), chord), 0)

    idx, w, j = spread(seg_link[inner] + 1)
    g = inner[w]
    r = 0.5 * width[path[g]]
    left = bend[g] > 0
    psi = end[g] + bend[g] * (j / (ribs[seg_link[g] + 1] - 1))
    rib = rib.index_put((idx,), both(pts[g + 1, 0], psi, torch.where(left, r, 0.0),
                                     torch.where(left, 0.0, r)))  # the outgoing segment's start
    for links, seg, at, turn0 in ((start_link, first, 0, math.pi), (end_link, last, 3, 0.0)):
        idx, w, j = spread(links)
        g = seg[w]
        psi = _angle(e[g, 0 if at == 0 else 2]) + turn0 + math.pi * (j / cap)
        r = 0.5 * width[path[g]]
        rib = rib.index_put((idx,), both(pts[g, at], psi, r, 0 * r))
    lead = off[start_link]  # a path's first rib has no chord
    count = off[end_link] + cap + 1 - lead
    length = length - torch.repeat_interleave(length[lead], count)
    return rib, length, length[lead + count - 1].detach()
