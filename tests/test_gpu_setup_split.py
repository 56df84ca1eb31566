"""Links per thread in the set-up follow the number of links (one where all CTAs run at once):
on both sides of each change of the split, every tuning writes the same ribs and offsets."""
import numpy as np
import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _polyline(n):
    rng = np.random.default_rng(n)
    p = np.cumsum(rng.integers(-40, 41, (n + 1, 2)), axis=0) / 4.0
    pts = np.zeros((n, 4, 2))
    pts[:, 0], pts[:, 1] = p[:-1], p[1:]
    return W.make_batch("polyline", np.full(n, W.LINE), pts, np.ones(n), [n], 6.0, W.JOIN_ROUND,
                        W.CAP_ROUND, dtheta_deg=40.0)


@pytest.mark.parametrize("waves", [1, 2])
@pytest.mark.parametrize("over", [False, True])
def test_every_split_at_the_edges_of_the_rule(waves, over):
    import torch
    import paper_2007_00308_gb300 as ps
    few, more = (ps.DeviceBatch(_polyline(n)).n_link for n in (10, 20))
    per = (more - few) // 10
    edge = 256 * 2 * waves * torch.cuda.get_device_properties(0).multi_processor_count
    n = (edge - (few - 10 * per)) // per + (1 if over else 0)
    db = ps.DeviceBatch(_polyline(n))
    assert (db.n_link > edge) == over and abs(db.n_link - edge) <= per
    want = None
    for links in (1, 2, 4):
        ctx = ps.Context()
        ctx.set_tuning(ps.PS_TUNE_SETUP_LINKS, links)
        out = ps.tessellate(ctx, db, ps.PS_PREC_MIXED)
        ref = ps.TessOutput(db.n_link, db.n_path, out.capacity)
        ps.ps_tessellate_strokes(ctx, db, ref, ps.PS_PREC_MIXED)
        assert ctx.status() == 0
        R = int(ref.n_rib.item())
        assert R == int(out.n_rib.item()) > n
        got = [getattr(ref, k)[:R] for k in ("rib", "tag", "s")] + [ref.link_rib_off, ref.path_len]
        assert bool((ref.link_rib_off[1:] >= ref.link_rib_off[:-1]).all())
        want = want or [t.clone() for t in got]
        for a, r in zip(got, want):
            assert torch.equal(a, r)
