"""Requantized bytes from strided convolutions on 128 and 256 filters or more: the fragment epilogue with its reordered weight
rows, output boxes staged in shared memory, and activations in tensor memory, all behind the im2col loader.  Every
output has to match the oracle bit for bit, and nothing is written past the end."""
import numpy as np
import pytest
import torch

import oracle
import sparq_synth as synth
import paper_2105_11010_b200 as sparq

NONE = sparq.SparqParams(sparq.MODE_NONE)
V5 = sparq.SparqParams()
V5_TRIM = sparq.SparqParams(sparq.MODE_VSPARQ, 4, 0x1F, sparq.ROUND_TRUNCATE)
V3OPT = sparq.SparqParams(sparq.MODE_VSPARQ, 4, 0x15, sparq.ROUND_NEAREST)
V7_TRIM = sparq.SparqParams(sparq.MODE_VSPARQ, 2, 0x7F, sparq.ROUND_TRUNCATE)
B6 = sparq.SparqParams(sparq.MODE_BSPARQ, 3, 0x3F, sparq.ROUND_NEAREST)
B5_TRIM = sparq.SparqParams(sparq.MODE_BSPARQ, 4, 0x1F, sparq.ROUND_TRUNCATE)

CASES = [
    # 256-wide tiles, a dozen and more steps: activations in tensor memory
    (25, 39, 1536, 256, 1, 2, V5, False), (25, 39, 1536, 224, 1, 2, V5_TRIM, False), (25, 39, 1792, 256, 1, 2, B5_TRIM, False),
    (25, 39, 1664, 256, 1, 2, V7_TRIM, False), (26, 39, 768, 480, 1, 2, V3OPT, False), (25, 39, 256, 256, 3, 2, B6, False),
    # 256-wide tiles, fragments straight to memory, with and without a residual
    (25, 39, 512, 256, 1, 2, V5, True), (25, 39, 512, 256, 1, 2, NONE, False), (25, 39, 384, 224, 1, 2, NONE, True), (25, 39, 128, 256, 3, 2, NONE, False), (25, 39, 1552, 256, 1, 2, B5_TRIM, False),
    # boxes through shared memory
    (26, 57, 64, 256, 1, 2, V5, False), (26, 57, 128, 288, 1, 2, V5_TRIM, True), (26, 57, 80, 256, 1, 2, NONE, True), (52, 57, 96, 128, 1, 2, B6, True), (52, 57, 64, 512, 1, 2, V5, True), (52, 57, 128, 512, 1, 2, NONE, False),
    # 128- and 64-wide tiles
    (26, 57, 256, 128, 1, 2, V5_TRIM, False), (26, 57, 64, 96, 3, 2, V5, True), (52, 57, 256, 64, 1, 2, V5, False)]


@pytest.mark.parametrize("nb,hw,c,cout,r,stride,p,residual", CASES)
def test_the_cases_go_through_the_im2col_loader(nb, hw, c, cout, r, stride, p, residual):
    assert sparq.sparq_selftest_form((nb, hw, hw, c), (cout, r, r, c), (stride, stride), (r // 2, r // 2), p) == sparq.FORM_FULL


@pytest.mark.gpu
@pytest.mark.parametrize("nb,hw,c,cout,r,stride,p,residual", CASES)
def test_bytes(nb, hw, c, cout, r, stride, p, residual):
    pad = r // 2
    x, w = synth.activations(c, (nb, hw, hw, c), 0.5), synth.weights(cout, (cout, r, r, c))
    scale, bias, inv = synth.scales(cout, cout), synth.bias(cout, cout), synth.inv_out_scale(r * r * c)
    acc = oracle.conv2d_nhwc(x, w, (stride, stride), (pad, pad), p.mode, p.window_bits, p.placement_mask, p.rounding)
    res = synth.activations(cout + 1, acc.shape, 0.5) if residual else None
    _, want = oracle.epilogue(acc, scale, bias, True, inv, residual=res, residual_scale=0.02)
    dev = [torch.from_numpy(t).cuda() for t in (x, w, scale, bias)]
    rd = torch.from_numpy(res).cuda() if residual else None
    for _ in range(3):
        out = torch.full((acc.size + 64,), 0xA5, dtype=torch.uint8, device="cuda")
        sparq.sparq_conv2d_nhwc_s8(dev[0], dev[1], (stride, stride), (pad, pad), p, scale=dev[2], bias=dev[3], relu=True, inv_out_scale=inv,
                                   u8_out=out[:acc.size].view(acc.shape), residual=rd, residual_scale=0.02)
        sparq.sparq_check()
        got = out.cpu().numpy()
        assert np.array_equal(got[:acc.size].reshape(acc.shape), want)
        assert (got[acc.size:] == 0xA5).all()
