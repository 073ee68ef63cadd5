"""Calls that run as transform into scratch memory + plain contraction."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import sparq_synth as synth
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


def test_a_captured_call_is_kernels_only():
    """Its graph can be cloned, added to another graph and instantiated more than once."""
    m, n, k = 1024 + 33, 4096, 4096
    A, B, p = synth.activations(5, (m, k), 0.5), synth.weights(5, (k, n)), sparq.SparqParams()
    Ad, Bd = torch.from_numpy(A).cuda(), torch.from_numpy(np.ascontiguousarray(B.T)).cuda()
    acc = torch.zeros((m, n), dtype=torch.int32, device="cuda")
    sparq.sparq_gemm_s8(Ad, Bd, p, acc_out=acc)
    sparq.sparq_check()
    rows = np.arange(0, m, 61)
    want = oracle.gemm(A[rows], B, p.mode, 4, 0x1F, 1)
    assert np.array_equal(acc.cpu().numpy()[rows], want)
    rt = ctypes.CDLL("libcudart.so.12")
    vp = ctypes.c_void_p
    stream = torch.cuda.Stream()
    st = vp(stream.cuda_stream)

    def ok(rc):
        assert rc == 0, rc

    graph, clone, parent, node = vp(), vp(), vp(), vp()
    ok(rt.cudaStreamBeginCapture(st, 0))
    sparq.sparq_gemm_s8(Ad, Bd, p, acc_out=acc, stream=stream)
    ok(rt.cudaStreamEndCapture(st, ctypes.byref(graph)))
    ok(rt.cudaGraphClone(ctypes.byref(clone), graph))
    ok(rt.cudaGraphCreate(ctypes.byref(parent), 0))
    ok(rt.cudaGraphAddChildGraphNode(ctypes.byref(node), parent, None, ctypes.c_size_t(0), graph))
    execs = [vp() for _ in range(4)]
    for e, g in zip(execs, (graph, graph, clone, parent)):
        ok(rt.cudaGraphInstantiate(ctypes.byref(e), g, ctypes.c_ulonglong(0)))
    for e in execs:
        acc.zero_()
        torch.cuda.synchronize()
        ok(rt.cudaGraphLaunch(e, st))
        stream.synchronize()
        assert np.array_equal(acc.cpu().numpy()[rows], want)
    for e in execs:
        ok(rt.cudaGraphExecDestroy(e))
    for g in (parent, clone, graph):
        ok(rt.cudaGraphDestroy(g))
    sparq.sparq_check()
