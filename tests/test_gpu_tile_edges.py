"""Kernels at the sizes where their tilings can go wrong, byte for byte against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import sparq_synth as synth
import paper_2105_11010_b200 as sparq

pytestmark = pytest.mark.gpu

# a warp encodes chunks of 128 units of 16 activations, two blocks of 16 warps per SM
CHUNKS_RESIDENT = 148 * 2 * 16


@pytest.mark.parametrize("n,mask", [(4, 0x1F), (4, 0x15), (4, 0x11), (3, 0x3F), (3, 0x35), (3, 0x29), (2, 0x7F), (2, 0x55)])
@pytest.mark.parametrize("mode,units", [(m, u) for m in (sparq.MODE_BSPARQ, sparq.MODE_VSPARQ) for u in (1, 127, 129)] +
                         [(sparq.MODE_VSPARQ, CHUNKS_RESIDENT * 128 + 131)])
def test_codec_chunks(n, mask, mode, units):
    x = synth.activations(units % 97, (units, 16), 0.5)
    p = sparq.SparqParams(mode, n, mask, 1)
    cb = sparq.sparq_packed_ctrl_bits(p)
    xg = torch.from_numpy(x).cuda()
    # guard bytes behind every plane: nothing may be written past its end
    data = torch.full((units * 2 * n + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    ctrl = torch.full((units * cb + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    out = torch.full((units * 16 + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    sparq.sparq_pack(xg, p, data, ctrl)
    sparq.sparq_unpack(data, ctrl, p, out[:units * 16].view(units, 16))
    sparq.sparq_check()
    wd, wc = oracle.pack_n(x, mode, n, mask, 1)
    for got, want in ((data, wd), (ctrl, wc), (out, oracle.transform(x, mode, n, mask, 1).reshape(-1))):
        got = got.cpu().numpy()
        assert np.array_equal(got[:-16], want.reshape(-1))
        assert (got[-16:] == 0xA5).all()


@pytest.mark.parametrize("mode", [sparq.MODE_NONE, sparq.MODE_VSPARQ])
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("n", [64, 96, 256, 288, 512])
def test_staged_output(mode, residual, n):
    """Requantized bytes through shared memory (short reductions, more tiles than SMs): row and column
    tails inside a box, a box wholly outside, several column tiles; nothing written past the end."""
    m, k = 148 * 128 * 2 + 128 * 5 + 45, 64
    A = synth.activations(n, (m, k), 0.5)
    B = synth.weights(n, (k, n))
    scale, bias, inv = synth.scales(n, n), synth.bias(n, n), synth.inv_out_scale(k)
    res = synth.activations(n + 1, (m, n), 0.5) if residual else None
    p = sparq.SparqParams(mode, 4, 0x1F, 1)
    out = torch.full((m * n + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    sparq.sparq_gemm_s8(torch.from_numpy(A).cuda(), torch.from_numpy(np.ascontiguousarray(B.T)).cuda(), p,
                        scale=torch.from_numpy(scale).cuda(), bias=torch.from_numpy(bias).cuda(), relu=True,
                        inv_out_scale=inv, u8_out=out, residual=torch.from_numpy(res).cuda() if residual else None,
                        residual_scale=0.02)
    sparq.sparq_check()
    acc = oracle.gemm(A, B, mode, 4, 0x1F, 1)
    _, want = oracle.epilogue(acc, scale, bias, True, inv, residual=res, residual_scale=0.02)
    got = out.cpu().numpy()
    assert np.array_equal(got[:m * n].reshape(m, n), want)
    assert (got[m * n:] == 0xA5).all()


@pytest.mark.parametrize("mode", [sparq.MODE_NONE, sparq.MODE_VSPARQ])
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("n,tail", [(160, 1), (224, 33), (256, 127), (480, 8)])
def test_wide_tiles_straight_to_memory(mode, residual, n, tail):
    """256-wide tiles of a long reduction (not staged): a warp's rows and 32-column groups at the tails of the
    matrix, and tiles with columns past N; nothing written past the end."""
    m, k = 148 * 128 + tail, 1024
    A = synth.activations(n, (m, k), 0.5)
    B = synth.weights(n, (k, n))
    scale, bias, inv = synth.scales(n, n), synth.bias(n, n), synth.inv_out_scale(k)
    res = synth.activations(n + 1, (m, n), 0.5) if residual else None
    p = sparq.SparqParams(mode, 4, 0x1F, 1)
    out = torch.full((m * n + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    sparq.sparq_gemm_s8(torch.from_numpy(A).cuda(), torch.from_numpy(np.ascontiguousarray(B.T)).cuda(), p,
                        scale=torch.from_numpy(scale).cuda(), bias=torch.from_numpy(bias).cuda(), relu=True,
                        inv_out_scale=inv, u8_out=out, residual=torch.from_numpy(res).cuda() if residual else None,
                        residual_scale=0.02)
    sparq.sparq_check()
    acc = oracle.gemm(A, B, mode, 4, 0x1F, 1)
    _, want = oracle.epilogue(acc, scale, bias, True, inv, residual=res, residual_scale=0.02)
    got = out.cpu().numpy()
    assert np.array_equal(got[:m * n].reshape(m, n), want)
    assert (got[m * n:] == 0xA5).all()


@pytest.mark.parametrize("mode,n,mask", [(sparq.MODE_VSPARQ, 4, 0x1F), (sparq.MODE_VSPARQ, 4, 0x15), (sparq.MODE_BSPARQ, 3, 0x3F), (sparq.MODE_VSPARQ, 2, 0x55)])
@pytest.mark.parametrize("m,cols,k", [(148 * 128 + 1, 160, 1040), (148 * 128 * 2 + 97, 256, 528), (148 * 128 - 31, 224, 1552)])
def test_activations_in_tensor_memory(mode, n, mask, m, cols, k):
    """256-wide tiles of long reductions: a last step that is mostly padding, more steps than either ring has
    stages by an odd number, several tiles per CTA on one accumulator, a last tile of a few rows."""
    A = synth.activations(k, (m, k), 0.5)
    B = synth.weights(cols, (k, cols))
    scale, bias, inv = synth.scales(cols, cols), synth.bias(cols, cols), synth.inv_out_scale(k)
    out = torch.full((m * cols + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    sparq.sparq_gemm_s8(torch.from_numpy(A).cuda(), torch.from_numpy(np.ascontiguousarray(B.T)).cuda(), sparq.SparqParams(mode, n, mask, 1),
                        scale=torch.from_numpy(scale).cuda(), bias=torch.from_numpy(bias).cuda(), relu=True, inv_out_scale=inv, u8_out=out)
    sparq.sparq_check()
    _, want = oracle.epilogue(oracle.gemm(A, B, mode, n, mask, 1), scale, bias, True, inv)
    got = out.cpu().numpy()
    assert np.array_equal(got[:m * cols].reshape(m, cols), want)
    assert (got[m * cols:] == 0xA5).all()


@pytest.mark.parametrize("mode,n", [(sparq.MODE_VSPARQ, 4), (sparq.MODE_BSPARQ, 3)])
def test_transform_first_gemm(mode, n):
    """Long reductions with many column tiles run as transform + plain contraction: two streams at
    once, each with scratch memory of its own, and again inside a captured graph."""
    m, cols, k = 1024 + 45, 2048, 1040
    mask = {4: 0x1F, 3: 0x3F}[n]
    p = sparq.SparqParams(mode, n, mask, 1)
    A = [synth.activations(70 + i, (m, k), 0.5) for i in range(2)]
    B = synth.weights(72, (k, cols))
    want = [oracle.gemm(a, B, mode, n, mask, 1) for a in A]
    Ad = [torch.from_numpy(a).cuda() for a in A]
    Bd = torch.from_numpy(np.ascontiguousarray(B.T)).cuda()
    out = [torch.zeros((m, cols), dtype=torch.int32, device="cuda") for _ in A]
    streams = [torch.cuda.Stream() for _ in A]
    torch.cuda.synchronize()
    for _ in range(3):
        for i, s in enumerate(streams):
            sparq.sparq_gemm_s8(Ad[i], Bd, p, acc_out=out[i], stream=s)
    for s in streams:
        sparq.sparq_check(s)
    for i in range(2):
        assert np.array_equal(out[i].cpu().numpy(), want[i])
    out[0].zero_()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=streams[0]):
        sparq.sparq_gemm_s8(Ad[0], Bd, p, acc_out=out[0])
    for _ in range(2):
        g.replay()
    sparq.sparq_check()
    assert np.array_equal(out[0].cpu().numpy(), want[0])


@pytest.mark.parametrize("c,cout,r,hw,nb,stride", [
    (48, 64, 5, 35, 3, 1),      # one partial 64-channel block, 25 resident taps, odd image
    (16, 40, 3, 56, 2, 1),      # mostly fill
    (80, 48, 3, 28, 2, 1),      # few filters on a partial 128-channel block
    (64, 128, 3, 28, 2, 1),     # half-empty 128-channel block
    (192, 192, 3, 17, 2, 1),    # two channel blocks, the second partial, streamed weights
    (144, 300, 3, 14, 40, 1),   # 256-wide tiles, partial block and partial column tile
    (512, 264, 3, 7, 20, 1),    # small maps: transform first, then im2col
    (256, 512, 3, 14, 9, 2),    # strided
])
@pytest.mark.parametrize("mode", [sparq.MODE_NONE, sparq.MODE_VSPARQ])
def test_conv_channel_blocks(c, cout, r, hw, nb, stride, mode):
    x = synth.activations(c + cout, (nb, hw, hw, c), 0.5)
    w = synth.weights(c + cout, (cout, r, r, c))
    p = sparq.SparqParams(mode, 4, 0x1F, 1)
    ho = (hw + 2 * (r // 2) - r) // stride + 1
    acc = torch.full((nb * ho * ho * cout + 16,), -7, dtype=torch.int32, device="cuda")
    sparq.sparq_conv2d_nhwc_s8(torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), (stride, stride), (r // 2, r // 2), p,
                               acc_out=acc)
    sparq.sparq_check()
    got = acc.cpu().numpy()
    want = oracle.conv2d_nhwc(x, w, (stride, stride), (r // 2, r // 2), mode, 4, 0x1F, 1)
    assert np.array_equal(got[:-16], want.reshape(-1))
    assert (got[-16:] == -7).all()


@pytest.mark.parametrize("m,n,k", [
    (1, 64, 2048),       # one row: most CTAs of a cluster of eight own nothing
    (49, 512, 2048),     # rows that do not divide over the cluster
    (64, 61, 576),       # one 64-row tile, ragged columns (scalar accesses), five steps
    (65, 264, 1040),     # a second tile of one row, a partial last reduction step
    (200, 72, 1024),     # partial last tile
    (333, 128, 16),      # one step: not shared
    (700, 136, 320),     # 64-byte steps
])
@pytest.mark.parametrize("mode", [sparq.MODE_NONE, sparq.MODE_VSPARQ])
@pytest.mark.parametrize("outputs", ["u8", "all"])
def test_few_tiles_gemm(m, n, k, mode, outputs):
    A = synth.activations(m + k, (m, k), 0.5)
    B = synth.weights(m + k, (k, n))
    scale, bias, inv = synth.scales(n, n), synth.bias(n, n), synth.inv_out_scale(k)
    res = synth.activations(m + n, (m, n), 0.5)
    p = sparq.SparqParams(mode, 4, 0x1F, 1)
    acc = oracle.gemm(A, B, mode, 4, 0x1F, 1)
    f32, u8 = oracle.epilogue(acc, scale, bias, True, inv, residual=res, residual_scale=0.02)
    d = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    guard = lambda dt, v: torch.full((m * n + 64,), v, dtype=dt, device="cuda")  # noqa: E731
    out = {"u8_out": guard(torch.uint8, 0xA5)}
    if outputs == "all":
        out.update(acc_out=guard(torch.int32, -7), f32_out=guard(torch.float32, -7.0))
    for _ in range(2):       # the second launch starts beside the first
        sparq.sparq_gemm_s8(d(A), d(np.ascontiguousarray(B.T)), p, scale=d(scale), bias=d(bias), relu=True, inv_out_scale=inv,
                            residual=d(res), residual_scale=0.02, **out)
    sparq.sparq_check()
    for name, want, fill in (("u8_out", u8, 0xA5), ("acc_out", acc, -7), ("f32_out", f32, -7.0)):
        if name in out:
            got = out[name].cpu().numpy()
            assert np.array_equal(got[:m * n].reshape(m, n), want), name
            assert (got[m * n:] == fill).all()


@pytest.mark.parametrize("nb,hw,c,cout,r,stride", [(1, 7, 512, 512, 3, 1), (1, 14, 256, 256, 3, 1), (1, 14, 144, 200, 3, 2),
                                                   (3, 9, 80, 130, 5, 1), (1, 28, 48, 512, 1, 2)])
@pytest.mark.parametrize("mode", [sparq.MODE_NONE, sparq.MODE_VSPARQ])
def test_few_tiles_conv(nb, hw, c, cout, r, stride, mode):
    x = synth.activations(c + cout, (nb, hw, hw, c), 0.5)
    w = synth.weights(c + cout, (cout, r, r, c))
    ho = (hw + 2 * (r // 2) - r) // stride + 1
    acc = torch.full((nb * ho * ho * cout + 16,), -7, dtype=torch.int32, device="cuda")
    sparq.sparq_conv2d_nhwc_s8(torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda(), (stride, stride), (r // 2, r // 2),
                               sparq.SparqParams(mode, 4, 0x1F, 1), acc_out=acc)
    sparq.sparq_check()
    got = acc.cpu().numpy()
    assert np.array_equal(got[:-16], oracle.conv2d_nhwc(x, w, (stride, stride), (r // 2, r // 2), mode, 4, 0x1F, 1).reshape(-1))
    assert (got[-16:] == -7).all()


@pytest.mark.parametrize("nb,hw,c,cout", [(7, 20, 64, 64), (7, 20, 128, 128), (11, 14, 256, 256), (37, 28, 128, 320)])
@pytest.mark.parametrize("kind", ["u8", "u8+residual", "all"])
@pytest.mark.parametrize("mode", [sparq.MODE_NONE, sparq.MODE_VSPARQ])
def test_window_output_kinds(nb, hw, c, cout, kind, mode):
    """3x3 convolutions on every window tile, for each kind of output that a kernel is instantiated for."""
    x, w = synth.activations(c, (nb, hw, hw, c), 0.5), synth.weights(c, (cout, 3, 3, c))
    scale, bias, inv = synth.scales(c, cout), synth.bias(c, cout), synth.inv_out_scale(9 * c)
    res = synth.activations(cout + 1, (nb * hw * hw, cout), 0.5) if "residual" in kind else None
    f32, u8 = oracle.epilogue(oracle.conv2d_nhwc(x, w, (1, 1), (1, 1), mode, 4, 0x1F, 1).reshape(-1, cout), scale, bias, True, inv,
                              residual=res, residual_scale=0.02)
    d = lambda v: torch.from_numpy(v).cuda()  # noqa: E731
    out = {"u8_out": torch.full((u8.size + 64,), 3, dtype=torch.uint8, device="cuda")}
    if kind == "all":
        out["f32_out"] = torch.full((u8.size + 64,), 3, dtype=torch.float32, device="cuda")
    sparq.sparq_conv2d_nhwc_s8(d(x), d(w), (1, 1), (1, 1), sparq.SparqParams(mode, 4, 0x1F, 1), scale=d(scale), bias=d(bias), relu=True,
                               inv_out_scale=inv, residual=None if res is None else d(res), residual_scale=0.02, **out)
    sparq.sparq_check()
    for name, want in (("u8_out", u8), ("f32_out", f32)):
        if name in out:
            got = out[name].cpu().numpy()
            assert np.array_equal(got[:u8.size].reshape(-1, cout), want), name
            assert (got[u8.size:] == 3).all()


@pytest.mark.parametrize("n", [1, 3, 31, 33, 61, 68, 72, 80, 127, 130, 200, 261])
@pytest.mark.parametrize("residual", [False, True])
def test_ragged_columns(n, residual):
    """Every row length modulo the store widths, in launches with several tiles per SM."""
    m, k = 148 * 128 * 2 + 77, 48
    A, B = synth.activations(n, (m, k), 0.5), synth.weights(n, (k, n))
    scale, bias, inv = synth.scales(n, n), synth.bias(n, n), synth.inv_out_scale(k)
    res = synth.activations(n + 1, (m, n), 0.5) if residual else None
    p = sparq.SparqParams(sparq.MODE_VSPARQ, 4, 0x1F, 1)
    acc = oracle.gemm(A, B, p.mode, 4, 0x1F, 1)
    f32, u8 = oracle.epilogue(acc, scale, bias, True, inv, residual=res, residual_scale=0.02)
    d = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    for names in (["u8_out"], ["acc_out", "f32_out", "u8_out"]):
        dt = {"u8_out": torch.uint8, "acc_out": torch.int32, "f32_out": torch.float32}
        out = {q: torch.full((m * n + 64,), 3, dtype=dt[q], device="cuda") for q in names}
        sparq.sparq_gemm_s8(d(A), d(np.ascontiguousarray(B.T)), p, scale=d(scale), bias=d(bias), relu=True, inv_out_scale=inv,
                            residual=d(res) if residual else None, residual_scale=0.02, **out)
        sparq.sparq_check()
        for q in names:
            got = out[q].cpu().numpy()
            assert np.array_equal(got[:m * n].reshape(m, n), {"u8_out": u8, "acc_out": acc, "f32_out": f32}[q]), q
            assert (got[m * n:] == 3).all()


@pytest.mark.parametrize("m,n,k", [(148 * 256 + 300, 128, 256), (148 * 256 * 2 + 45, 104, 144), (148 * 128 + 31, 61, 528),
                                   (148 * 256 + 1, 264, 96)])
@pytest.mark.parametrize("nb,mask,rnd", [(4, 0x1F, 1), (4, 0x1F, 0), (4, 0x15, 1), (3, 0x3F, 1), (2, 0x7F, 0)])
def test_sparse24_fused(m, n, k, nb, mask, rnd):
    """Expansion inside the product: partial row tiles, partial reduction steps, ragged columns."""
    A = synth.activations(m % 91, (m, k), 0.5)
    vals, pos = synth.sparse24_weights(n, n, k)
    p = sparq.SparqParams(sparq.MODE_VSPARQ, nb, mask, rnd)
    kx = sparq.sparq_sparse24_expanded_k(k, p)
    d = lambda x: torch.from_numpy(x).cuda()  # noqa: E731
    w = torch.empty((n, kx), dtype=torch.int8, device="cuda")
    sparq.sparq_sparse24_expand_weights(d(vals), d(pos), p, w)
    acc = torch.full((m * n + 16,), -7, dtype=torch.int32, device="cuda")
    sparq.sparq_gemm_s8_sparse24(d(A), w, p, workspace=torch.empty(m * kx, dtype=torch.uint8, device="cuda"), acc_out=acc)
    sparq.sparq_check()
    got = acc.cpu().numpy()
    rows = np.unique(np.concatenate([np.arange(0, m, 997), np.arange(300), np.arange(m - 300, m)]))
    want = oracle.gemm_sparse24(A[rows], vals, pos, p.mode, nb, mask, rnd)
    assert np.array_equal(got[:-16].reshape(m, n)[rows], want)
    assert (got[-16:] == -7).all()


@pytest.mark.parametrize("cout,k", [(1, 4), (3, 5), (7, 1020), (5, 5120), (4, 5124), (3, 9001), (130, 64)])
def test_quantize_weight_rows(cout, k):
    """Row lengths around what a block keeps in registers, with and without whole vectors."""
    w = np.random.default_rng(cout + k).standard_normal((cout, k)).astype(np.float32)
    w[0, 0] = np.nan
    out = torch.full((cout * k + 16,), 99, dtype=torch.int8, device="cuda")
    sc = torch.zeros(cout, device="cuda")
    sparq.sparq_quantize_weight_s8(torch.from_numpy(w).cuda(), out, sc)
    want_q, want_s = oracle.quantize_weight(w)
    got = out.cpu().numpy()
    assert np.array_equal(got[:-16].reshape(cout, k), want_q) and (got[-16:] == 99).all()
    assert np.array_equal(sc.cpu().numpy(), want_s)


@pytest.mark.parametrize("n", [7, 4096, (64 << 20) // 4 + 4096 * 3 + 5])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_calibration_passes(n, dtype):
    """Maximum and quantization of one tensor, beyond the part that the first pass leaves in L2."""
    x = torch.randn(n, device="cuda").to(dtype)
    mx, q = torch.zeros(1, device="cuda"), torch.full((n + 16,), 7, dtype=torch.uint8, device="cuda")
    sparq.sparq_absmax(x, mx)
    sparq.sparq_quantize_act_u8(x, mx, q)
    xh = x.float().cpu().numpy()
    assert mx.item() == oracle.absmax(xh)
    got = q.cpu().numpy()
    assert np.array_equal(got[:n], oracle.quantize_act(xh, mx.item())) and (got[n:] == 7).all()


@pytest.mark.parametrize("rows,row_len", [(1, 17), (1, 31), (5, 17), (64, 19), (333, 33), (7, 4097), (1000, 1023), (3, 15), (257, 101)])
@pytest.mark.parametrize("n,mask,rnd", [(4, 0x1F, 1), (4, 0x1F, 0), (4, 0x15, 1), (3, 0x3F, 1), (3, 0x29, 0), (2, 0x7F, 0)])
def test_transform_odd_rows(rows, row_len, n, mask, rnd):
    """Row boundaries at every place of a vector, a last partial vector, and in place."""
    x = synth.activations(rows + row_len, (rows, row_len), 0.4)
    p = sparq.SparqParams(sparq.MODE_VSPARQ, n, mask, rnd)
    want = oracle.transform(x, p.mode, n, mask, rnd).reshape(-1)
    xd = torch.from_numpy(x).cuda().reshape(-1)
    out = torch.full((x.size + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    sparq.sparq_quantize(xd, out, rows, row_len, p)
    got = out.cpu().numpy()
    assert np.array_equal(got[:-16], want) and (got[-16:] == 0xA5).all()
    sparq.sparq_quantize(xd, xd, rows, row_len, p)
    assert np.array_equal(xd.cpu().numpy(), want)
