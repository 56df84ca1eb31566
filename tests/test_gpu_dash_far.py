"""Dash pieces far along a path, to the bit: patterns off every binary grid, arc lengths out to
2^18 periods, where the prefilter's and the pair walk's error bounds rest on every product and
sum being rounded by itself."""
import numpy as np
import pytest

import oracle
from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (the last two patterns are multiples of a binary grid: decided without a margin)
PATTERNS = [("-1.7", "7.3 2.1"), ("0.01", "0.1 0.2 0.3 0.05"), ("0", "1e-3 2e-3"),
            ("1e6", "2.5 1.25 0.3"), ("0", "12 6"), ("3.25", "9 3 1 3")]


@pytest.mark.parametrize("capped", [False, True])
@pytest.mark.parametrize("offset,pattern", PATTERNS)
def test_far_dashes_match_oracle(offset, pattern, capped):
    import torch
    import paper_2007_00308_gb300 as ps
    pat = np.array(pattern.split(), np.float32)
    off = float(np.float32(offset))
    period = pat.astype(np.float64).sum()
    rng = np.random.default_rng(5)
    n = 200000
    # one quad per link: from 0 to 2^18 periods in, 2^-12 to 4 periods long, some of no length,
    # some that begin or end next to a stretch end
    cum = np.concatenate([[0.0], np.cumsum(pat.astype(np.float64))])
    sa = np.exp2(rng.uniform(-6, 18, n)) * period
    at = np.floor(sa / period) * period + cum[rng.integers(0, len(cum), n)] - off
    sa = np.maximum(np.where(rng.random(n) < 0.3, at + period * rng.uniform(-1e-5, 1e-5, n), sa), 0)
    sa = sa.astype(np.float32)
    ln = np.where(rng.random(n) < 0.1, 0.0, np.exp2(rng.uniform(-12, 2, n)) * period)
    sb = np.maximum((sa + ln).astype(np.float32), sa)
    s = np.stack([sa, sb], 1).reshape(-1)
    tag = np.tile(np.array([3, 2], np.uint32), n)
    rib = rng.uniform(-50, 4100, (2 * n, 4)).astype(np.float32)
    path_cap = np.array([W.CAP_SQUARE], np.uint8)
    dtheta = np.radians(10.0)
    want = (oracle.dash_capped(rib, s, tag, pat, off, path_cap, dtheta) if capped
            else oracle.dash(rib, s, tag, pat, off))
    m = len(want["s"])
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    z = lambda *shape, dt: torch.zeros(shape, dtype=dt, device="cuda")  # noqa: E731
    got = [z(m, 4, dt=torch.float32), z(m, dt=torch.float32), z(m, dt=torch.int32),
           z(m, dt=torch.int32), z(1, dt=torch.int64)]
    ctx = ps.Context()
    src = (d(rib), d(s), d(tag.view(np.int32)), d(np.array([2 * n], np.int64)), 2 * n, pat, off)
    if capped:
        ps.ps_dash_capped(ctx, *src, d(path_cap), float(np.float32(dtheta)), *got, m)
    else:
        ps.ps_dash(ctx, *src, *got, m)
    torch.cuda.synchronize()
    assert int(got[4].item()) == m
    assert ctx.status() == 0
    otag = got[2].cpu().numpy().view(np.uint32)
    assert np.array_equal(otag, want["tag"])
    assert np.array_equal(got[3].cpu().numpy(), want["src"])
    assert np.array_equal(got[1].cpu().numpy(), want["s"].astype(np.float32))
    piece = (otag & 2) == 2  # the caps' own vertices have a bound of their own elsewhere
    assert np.array_equal(got[0].cpu().numpy()[piece], want["rib"][piece].astype(np.float32))
