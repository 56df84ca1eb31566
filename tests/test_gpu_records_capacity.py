"""Ribs from a caller's records into buffers that are too small: the capacity error of the call it
stands for, and the ribs that fit."""
import ctypes

import pytest

from paper_2007_00308_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("short", [0, 1, 5000, None])
def test_capacity_of_the_records_call(short):
    import torch
    import paper_2007_00308_gb300 as ps
    L, P = ps.lib(), ctypes.c_void_p
    ctx, db = ps.Context(), ps.DeviceBatch(W.c2_batching(n_paths=9))
    want = ps.tessellate(ps.Context(), db, ps.PS_PREC_MIXED)
    R = int(want.n_rib.item())
    capacity = 0 if short is None else R - short
    out = ps.TessOutput(db.n_link, db.n_path, max(capacity, 1))
    seg, paths = db._structs()
    o = out._struct()
    o.capacity = capacity
    records = torch.empty(L.ps_record_bytes(db.n_link), dtype=torch.uint8, device="cuda")
    n = ctypes.c_int64(0)
    stream = P(torch.cuda.current_stream().cuda_stream)
    assert L.ps_link_records_sync(ctx.handle, ctypes.byref(seg), ctypes.byref(paths), db.dtheta,
                                  ps.PS_PREC_MIXED, ctypes.byref(o), P(records.data_ptr()), stream,
                                  ctypes.byref(n)) == 0
    assert n.value == R and ctx.status() == 0
    assert L.ps_emit_records(ctx.handle, ctypes.byref(seg), ctypes.byref(paths), ps.PS_PREC_MIXED,
                             ps.PS_TESS_ARCLENGTH, ctypes.byref(o), P(records.data_ptr()), stream) == 0
    assert ctx.status() == (ps.PS_ERR_CAPACITY if capacity < R else 0)
    assert torch.equal(out.rib[:capacity], want.rib[:capacity])
    assert torch.equal(out.s[:capacity], want.s[:capacity])
