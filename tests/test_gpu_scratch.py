"""Calls that run as transform into scratch memory + plain contraction."""
import pytest
import torch

import paper_2105_11010_b200 as sparq

pytestmark = pytest.mark.gpu

M, N, K = 1 << 18, 1028, 2048      # the transform alone takes 0.15 ms


@pytest.mark.parametrize("entry", ["gemm", "conv", "sparse24"])
@pytest.mark.parametrize("bad", ["placement", "columns", "no bytes"])
def test_a_refused_call_enqueues_nothing(entry, bad):
    n = N - 1 if bad == "columns" else N
    nxt = sparq.SparqParams(sparq.MODE_VSPARQ, 4, 0x0F if bad == "placement" else 0x1F, 1)
    out = {"f32_out" if bad == "no bytes" else "u8_out": torch.empty(M * n, dtype=torch.float32 if bad == "no bytes" else torch.uint8, device="cuda")}
    a, w = torch.zeros((M, K), dtype=torch.uint8, device="cuda"), torch.zeros((n, K), dtype=torch.int8, device="cuda")
    p, scale = sparq.SparqParams(), torch.ones(n, device="cuda")
    call = {
        "gemm": lambda q, **kw: sparq.sparq_gemm_s8(a, w, q, scale=scale, **kw),
        "conv": lambda q, **kw: sparq.sparq_conv2d_nhwc_s8(a.view(64, 64, 64, K), w.view(n, 1, 1, K), (1, 1), (0, 0), q, scale=scale, **kw),
    }
    if entry == "sparse24":            # its wrapper passes no next_transform on
        native = sparq.load_native()
        w3, ws = torch.zeros((n, 3 * 64), dtype=torch.int8, device="cuda"), torch.empty(M * 3 * 64, dtype=torch.uint8, device="cuda")
        a64 = a.view(-1)[:M * 64].view(M, 64)
        args = [out.get(k) for k in ("acc_out", "f32_out", "u8_out")]
        torch.cuda.synchronize()
        rc = native.gemm_sparse24(a64, w3, p, ws, scale, None, False, 1.0, *args, nxt, None, 0.0, None)
        idle = torch.cuda.current_stream().query()
        assert rc < 0
    else:
        call[entry](sparq.SparqParams(sparq.MODE_NONE), **out)     # everything lazy has been set up
        torch.cuda.synchronize()
        with pytest.raises(sparq.SparqError):
            call[entry](p, next_transform=nxt, **out)
        idle = torch.cuda.current_stream().query()
    assert idle, "the refused call has enqueued work"
    sparq.sparq_check()
