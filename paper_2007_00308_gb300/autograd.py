"""torch.autograd.Function over the tessellation: (control points, widths) ->
(rib vertices, cumulative arc length), with the library's adjoint kernel for
the backward pass.  Step counts are those of the forward pass."""
from __future__ import annotations

import torch

from . import (PS_PREC_MIXED, Context, DeviceBatch, _backward_records, _tessellate_exact,
               ps_tessellate_backward, tessellate)


def _in_memory(grad, like):
    """Whether the tensor's memory holds its values as ``like``'s would."""
    return (grad.layout == torch.strided and grad.dtype == like.dtype and grad.device == like.device
            and not grad.is_neg() and not grad._is_zerotensor())


def _upstream(grad, like, n):
    """The gradient of the first n rows of ``like`` as the adjoint reads it: dense,
    16-byte aligned, as long as ``like``."""
    if grad is not None and n == like.shape[0] and _in_memory(grad, like):
        grad = grad.contiguous()
        return grad if grad.data_ptr() % 16 == 0 else grad.clone()
    full = torch.zeros(like.shape, dtype=torch.float32, device=like.device)
    if grad is not None:
        full[:n] = grad
    return full


class PolarStroke(torch.autograd.Function):
    @staticmethod
    def forward(ctx, pts, width, batch, precision=PS_PREC_MIXED, psctx=None):
        """pts: float32 [S, 4, 2] on the GPU; width: float32 [P]; batch: the
        StrokeBatch giving types, weights, path structure, joins, caps and dtheta.
        Returns rib [R, 4] (N.x N.y P.x P.y) and s [R].  Until the backward pass the
        graph holds the ribs and t, and the links' records of 244 bytes each (65 MB
        for 4,096 paths of 32 segments)."""
        c = psctx or Context()
        db = DeviceBatch(batch, device=pts.device, seg_pts=pts.detach().contiguous().reshape(-1),
                         path_width=width.detach().contiguous(), wait=False)
        if db.n_path > 0:
            out, records, R = _tessellate_exact(c, db, precision, want_t=True)
        else:
            out, records, R = tessellate(c, db, precision, want_t=True), None, 0
        ctx.state = (c, db, out, records, precision)
        ctx.shapes = (pts.shape, width.shape)
        return out.rib[:R], out.s[:R]

    @staticmethod
    def backward(ctx, grad_rib, grad_s):
        c, db, out, records, precision = ctx.state
        R = grad_rib.shape[0] if grad_rib is not None else grad_s.shape[0]
        g_rib = _upstream(grad_rib, out.rib, R)
        g_s = _upstream(grad_s, out.s, R)
        g_pts = torch.empty(db.n_seg * 8, dtype=torch.float32, device=out.rib.device)
        g_w = torch.empty(db.n_path, dtype=torch.float32, device=out.rib.device)
        if records is not None:  # the forward's links, not set up again
            _backward_records(c, db, out, records, g_rib, g_s, g_pts, g_w, precision)
        else:
            ps_tessellate_backward(c, db, out, g_rib, g_s, g_pts, g_w, precision)
        return g_pts.reshape(ctx.shapes[0]), g_w.reshape(ctx.shapes[1]), None, None, None
