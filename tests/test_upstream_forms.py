"""Upstream gradients whose memory does not hold their values (lazily negated, all-zero without
storage, another type) reach the adjoint as dense FP32 values; plain ones in place."""
import numpy as np
import pytest
import torch

from paper_2007_00308_gb300.autograd import _upstream

LIKE = torch.empty((6, 4))


def _values(shape, dtype=torch.float32):
    return torch.arange(float(np.prod(shape)), dtype=dtype).reshape(shape) - 5.5


@pytest.mark.parametrize("form", ["negated", "negated column", "zero", "double", "plain"])
def test_memory_holds_the_values(form):
    if form == "negated":
        grad = torch._neg_view(_values((6, 4)))
    elif form == "negated column":
        grad = torch.view_as_complex(_values((6, 4, 2))).conj().imag
    elif form == "zero":
        grad = torch._efficientzerotensor((6, 4))
    else:
        grad = _values((6, 4), torch.float64 if form == "double" else torch.float32)
    want = grad.clone().resolve_neg().numpy().astype(np.float32) if form != "zero" else np.zeros((6, 4))
    got = _upstream(grad, LIKE, 6)
    assert got.dtype == torch.float32 and got.shape == LIKE.shape and got.is_contiguous()
    assert got.data_ptr() % 16 == 0 and got.data_ptr() != 0
    # what a kernel reads there
    read = np.ctypeslib.as_array((np.ctypeslib.ctypes.c_float * 24).from_address(got.data_ptr()))
    assert np.array_equal(read.reshape(6, 4), want)
    if form == "plain":
        assert got.data_ptr() == grad.data_ptr() or grad.data_ptr() % 16
