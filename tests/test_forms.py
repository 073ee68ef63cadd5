"""Which form a layer takes (a host-side rule on sizes and transform), and every form's results."""
import numpy as np
import pytest
import torch

import oracle
import sparq_synth as synth
import paper_2105_11010_b200 as sparq

V5 = sparq.SparqParams()
V6 = sparq.SparqParams(sparq.MODE_VSPARQ, 3, sparq.SET_6OPT, sparq.ROUND_NEAREST)
V7 = sparq.SparqParams(sparq.MODE_VSPARQ, 2, sparq.SET_7OPT, sparq.ROUND_NEAREST)
R35 = sparq.SparqParams(sparq.MODE_VSPARQ, 3, 0x35, sparq.ROUND_NEAREST)
R55 = sparq.SparqParams(sparq.MODE_VSPARQ, 2, 0x55, sparq.ROUND_NEAREST)
NONE = sparq.SparqParams(sparq.MODE_NONE)


def form(n, hw, c, cout, r, stride, p):
    return sparq.sparq_selftest_form((n, hw, hw, c), (cout, r, r, c), (stride, stride), (r // 2, r // 2), p)


@pytest.mark.parametrize("n,hw,c,cout,r,stride,p,want", [
    # few tiles: clusters on one tile where that is the faster form, and only there
    (1, 14, 256, 256, 3, 1, V5, sparq.FORM_SMALL),
    (1, 7, 512, 512, 3, 1, V5, sparq.FORM_SMALL),
    (8, 14, 512, 512, 5, 1, V5, sparq.FORM_WINDOW_STREAMED),
    (8, 17, 256, 512, 5, 1, V5, sparq.FORM_WINDOW_STREAMED),
    (17, 14, 384, 128, 7, 1, V6, sparq.FORM_WINDOW_STREAMED),
    (1, 28, 512, 64, 3, 1, V5, sparq.FORM_SMALL),
    # half-empty channel blocks
    (64, 17, 64, 256, 3, 1, V5, sparq.FORM_FULL),
    (128, 17, 32, 256, 3, 1, NONE, sparq.FORM_FULL),
    (17, 35, 48, 64, 5, 1, V5, sparq.FORM_WINDOW_RESIDENT),
    # windows that just fit beside a ring of two stages
    (64, 35, 384, 192, 3, 1, V6, sparq.FORM_WINDOW_STREAMED),
    (16, 56, 256, 64, 5, 1, R35, sparq.FORM_TRANSFORM_FIRST),
    # resident weights
    (128, 28, 128, 128, 3, 1, V5, sparq.FORM_WINDOW_RESIDENT),
    (32, 56, 64, 64, 3, 1, V5, sparq.FORM_WINDOW_RESIDENT),
    # 1x1 and strided layers
    (64, 56, 64, 256, 1, 1, V5, sparq.FORM_FULL),
    (1, 14, 1024, 256, 1, 1, V5, sparq.FORM_SMALL),
    (64, 7, 512, 512, 3, 1, V5, sparq.FORM_TRANSFORM_FIRST),
    (64, 14, 512, 512, 3, 2, V5, sparq.FORM_TRANSFORM_FIRST),
    (64, 7, 512, 512, 3, 1, NONE, sparq.FORM_FULL),
])
def test_form(n, hw, c, cout, r, stride, p, want):
    assert form(n, hw, c, cout, r, stride, p) == want


@pytest.mark.parametrize("n,hw", [(64, 56), (16, 112)])
@pytest.mark.parametrize("cout", [264, 320, 384])
def test_form_is_judged_by_the_tiles_it_is_launched_with(n, hw, cout):
    """80 channels: the launch chose its tile width by one 128-byte step per tap, where two 64-byte ones choose
    another.  Judged by that other one these layers were transformed first and took up to a quarter longer."""
    assert form(n, hw, 80, cout, 3, 2, V5) == sparq.FORM_FULL


@pytest.mark.parametrize("n,hw,c,cout,r,p,want", [
    # what a transform costs: 3- and 2-bit windows with the pair rule nearly twice that of 4-bit ones
    (5151, 1, 2608, 1680, 1, V7, sparq.FORM_TRANSFORM_FIRST), (4335, 1, 2160, 1352, 1, V6, sparq.FORM_TRANSFORM_FIRST),
    (1433, 1, 2944, 1896, 1, V7, sparq.FORM_TRANSFORM_FIRST), (12172, 1, 544, 1840, 1, V6, sparq.FORM_TRANSFORM_FIRST),
    # what a row costs through an im2col map: no less in 64-byte blocks, more where the last block is not full
    (8, 44, 48, 488, 5, V5, sparq.FORM_FULL), (6, 56, 432, 288, 3, V5, sparq.FORM_FULL), (3, 56, 272, 488, 3, V5, sparq.FORM_FULL),
    (10, 48, 336, 256, 3, V5, sparq.FORM_FULL)])
def test_form_follows_the_costs_of_transform_and_fetch(n, hw, c, cout, r, p, want):
    """Layers that took 10 to 40 % longer in the other form."""
    assert form(n, hw, c, cout, r, 1, p) == want


def test_form_refuses_bad_geometry():
    with pytest.raises(sparq.SparqError):
        sparq.sparq_selftest_form((1, 8, 8, 24), (16, 3, 3, 24), (1, 1), (1, 1), V5)
    with pytest.raises(sparq.SparqError):
        sparq.sparq_selftest_form((1, 2, 2, 16), (16, 5, 5, 16), (1, 1), (0, 0), V5)


@pytest.mark.gpu
@pytest.mark.parametrize("want,n,hw,c,cout,r,stride", [
    (sparq.FORM_TRANSFORM_FIRST, 31, 7, 512, 1032, 3, 1),
    (sparq.FORM_TRANSFORM_FIRST, 40, 14, 512, 712, 3, 2),
    (sparq.FORM_TRANSFORM_FIRST, 1, 33, 4096, 4104, 1, 1),
    (sparq.FORM_WINDOW_STREAMED, 5, 17, 256, 200, 5, 1),
    (sparq.FORM_WINDOW_STREAMED, 33, 14, 256, 264, 3, 1),
    (sparq.FORM_WINDOW_STREAMED, 40, 35, 384, 192, 3, 1),
    (sparq.FORM_WINDOW_RESIDENT, 9, 35, 96, 72, 3, 1),
    (sparq.FORM_SMALL, 2, 14, 320, 136, 3, 1),
    (sparq.FORM_FULL, 33, 17, 48, 264, 3, 1),
])
@pytest.mark.parametrize("p", [V5, V6], ids=["5opt", "6opt"])
@pytest.mark.parametrize("kind", ["acc", "u8+residual"])
def test_results_of_a_form(want, n, hw, c, cout, r, stride, p, kind):
    """All outputs against a contraction of the oracle's transform in float64 (integers: exact)."""
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert form(n, hw, c, cout, r, stride, p) == want
    x, w = synth.activations(c, (n, hw, hw, c), 0.5), synth.weights(cout, (cout, r, r, c))
    pad = r // 2
    d = lambda t: torch.from_numpy(t).cuda()  # noqa: E731
    t = oracle.transform(x.reshape(-1, c), p.mode, p.window_bits, p.placement_mask, p.rounding).reshape(x.shape)
    acc = torch.nn.functional.conv2d(d(t).permute(0, 3, 1, 2).double(), d(w).permute(0, 3, 1, 2).double(), stride=stride, padding=pad)
    acc = acc.permute(0, 2, 3, 1).reshape(-1, cout).round().to(torch.int32).cpu().numpy()
    if kind == "acc":
        out = torch.full((acc.size + 16,), -7, dtype=torch.int32, device="cuda")
        sparq.sparq_conv2d_nhwc_s8(d(x), d(w), (stride, stride), (pad, pad), p, acc_out=out)
        want_out, fill = acc, -7
    else:
        scale, bias, inv = synth.scales(cout, cout), synth.bias(cout, cout), synth.inv_out_scale(r * r * c)
        res = synth.activations(cout + 1, acc.shape, 0.5)
        _, want_out = oracle.epilogue(acc, scale, bias, True, inv, residual=res, residual_scale=0.02)
        out, fill = torch.full((acc.size + 16,), 3, dtype=torch.uint8, device="cuda"), 3
        sparq.sparq_conv2d_nhwc_s8(d(x), d(w), (stride, stride), (pad, pad), p, scale=d(scale), bias=d(bias), relu=True, inv_out_scale=inv,
                                   residual=d(res), residual_scale=0.02, u8_out=out)
    sparq.sparq_check()
    got = out.cpu().numpy()
    assert np.array_equal(got[:acc.size].reshape(acc.shape), want_out)
    assert (got[acc.size:] == fill).all()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 3, 4, 7, 12, 20, 28, 36, 52, 60, 65, 76])
@pytest.mark.parametrize("m,k", [(130, 48), (300, 1600)])
def test_few_tiles_narrow_columns(n, m, k):
    """Column counts whose groups of four do not divide the workers; one CTA a tile, and several."""
    A, B = synth.activations(n, (m, k), 0.5), synth.weights(n, (k, n))
    scale, bias, inv = synth.scales(n, n), synth.bias(n, n), synth.inv_out_scale(k)
    res = synth.activations(n + 1, (m, n), 0.5)
    acc = oracle.gemm(A, B, V5.mode, 4, 0x1F, 1)
    f32, u8 = oracle.epilogue(acc, scale, bias, True, inv, residual=res, residual_scale=0.02)
    d = lambda t: torch.from_numpy(t).cuda()  # noqa: E731
    out = {q: torch.full((m * n + 64,), 3, dtype=t, device="cuda") for q, t in
           (("acc_out", torch.int32), ("f32_out", torch.float32), ("u8_out", torch.uint8))}
    sparq.sparq_gemm_s8(d(A), d(np.ascontiguousarray(B.T)), V5, scale=d(scale), bias=d(bias), relu=True, inv_out_scale=inv,
                        residual=d(res), residual_scale=0.02, **out)
    sparq.sparq_check()
    for name, want in (("acc_out", acc), ("f32_out", f32), ("u8_out", u8)):
        got = out[name].cpu().numpy()
        assert np.array_equal(got[:m * n].reshape(m, n), want), name
        assert (got[m * n:] == 3).all()
