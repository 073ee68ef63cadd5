"""Sizes beyond the kernels' and the call module's integers are refused, on the host."""
import ctypes

import pytest
import torch

import paper_2105_11010_b200 as sparq
from paper_2105_11010_b200._binding import _CEpilogue


@pytest.mark.parametrize("n,h,w,r,stride", [(1 << 11, 1 << 10, (1 << 10) + 1, 1, 1), (1 << 12, 1 << 11, 1 << 10, 3, 1), (1 << 14, 1 << 10, 1 << 10, 3, 2)])
def test_too_many_output_pixels(n, h, w, r, stride):
    L, p = sparq.load_library(), sparq.SparqParams()._c()
    one = ctypes.c_void_p(1 << 20)          # never read: the call is refused before it touches a device
    e = _CEpilogue(scale=1 << 20, u8_out=1 << 20, inv_out_scale=1.0)
    rc = L.sparq_conv2d_nhwc_s8(one, n, h, w, 16, one, 16, r, r, stride, stride, r // 2, r // 2, ctypes.byref(p), ctypes.byref(e), None)
    assert rc == -2 and "output pixels" in sparq.sparq_last_error()


@pytest.mark.parametrize("rows,row_len", [(1 << 32, 1 << 32), (1 << 33, 1 << 31), (-1, -1), (-4, 16), (3, 16)])
def test_rows_and_row_length_beyond_the_tensor(rows, row_len):
    x = torch.zeros(32, dtype=torch.uint8)
    with pytest.raises(ValueError):
        sparq.sparq_quantize_host(x, x, rows, row_len, sparq.SparqParams())
