"""Every kernel that may start before its predecessor on the stream has finished waits for it before
it touches the caller's memory: weights included, whatever wrote them (this library's own weight
expansion, another library's kernel, a copy)."""
import os
import re

import numpy as np
import pytest
import torch

import oracle
import sparq_synth as synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_11010_b200", "csrc")
READS = re.compile(r"\b(tma_load\w*|tma_store\w*|ld16|ld_stream\w*|st_stream\w*|__ldg|__ldcs|__stcs|ld_global_v8|st_global_v8|issue_\w+)\s*\(")


def without_lambdas(text):
    """The text without the bodies of lambdas, which run where they are called."""
    out, i = "", 0
    for m in re.finditer(r"auto \w+ = \[&\][^{;]*\{", text):
        if m.start() < i:
            continue
        out += text[i:m.start()]
        depth, j = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        i = j
    return out + text[i:]


def kernels():
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\s*\([^;{]*\)\s*\{", text):
            body = text[m.end():text.find("__global__", m.end()) if "__global__" in text[m.end():] else len(text)]
            if "dep_wait();" in body:
                yield f, m.group(1), body


def block_end(text, i):
    """Index behind the block whose opening brace is at text[i]."""
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
    return j


def kernel_bodies():
    """kernels() with each body ending where it does."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\s*\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\([^;{]*\)\s*\{", text):
            body = text[m.end():block_end(text, m.end() - 1)]
            if "dep_wait();" in body:
                yield f, m.group(1), body


def roles(body):
    """(set-up, branches): the branches of the if / else-if chain over the warp's number that a kernel with several
    roles consists of (its longest such chain), and the text before it.  A kernel without one is all set-up."""
    best = (body, [])
    for m in re.finditer(r"\n    if (?=\([^{]*\bwarp\b)", body):
        chain, i = [], m.end()
        while True:
            a = body.index("{", i)
            i = block_end(body, a)
            chain.append(body[a:i])
            more = re.match(r"\s*else(?: if (?=\()| (?=\{))", body[i:])
            if not more:
                break
            i += more.end()
        if len(chain) > max(2, len(best[1])):
            best = (body[:m.start()], chain)
    return best


def test_bounded_waits_do_not_count_the_kernel_before():
    """A wait for a barrier gives up after about a second.  Where a role has not waited for the kernel before, one that
    releases its successor early and then takes long would use that time up: an expired EARLY wait first waits for
    that kernel and starts its clock again, once."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "sparq_gemm_kernel.cuh")).read())
    wait = text[text.index("bool mbar_wait("):]
    wait = wait[:block_end(wait, wait.index("{"))]
    a = wait.index("{", wait.index("if (clock64() - t0 > limit_cycles)"))
    expired = wait[a + 1:block_end(wait, a) - 1]
    again = re.match(r"\s*if \(!alone\) \{(.*?)\}", expired, re.S)
    assert again and [s.strip() for s in again.group(1).split(";")] == ["dep_wait()", "alone = true", "t0 = clock64()", "continue", ""]
    assert "*abort_flag = 1u;" in expired[again.end():] and "bool alone = !EARLY;" in wait
    # Waits of the roles that have not waited for the kernel before, in order: what their first operands land on or
    # come from is EARLY.  (Barriers that start free are waited for from a stage's second use on.)
    early = {}
    for f, name, body in kernel_bodies():
        setup, branches = roles(body)
        assert "mbar_wait" not in setup, name
        for i, role in enumerate(branches):
            waits = [m for m in re.finditer(r"mbar_wait(?:<([^>]*)>)?\((?:smem_u32\(&)?(\w+)", role) if not re.search("empty|done", m.group(2))]
            if "dep_wait();" not in role[:waits[0].start()]:
                early[name, i] = [(m.group(2), m.group(1)) for m in waits]
    streamed = "!B_RESIDENT"
    assert early == {
        ("sparq_gemm_kernel", 1): [("bar_full", "true"), ("bar_xf", "true"), ("bar_full", None)],
        ("sparq_gemm_kernel", 3): [("bar_raw", "true"), ("bar_full", "true")],
        # resident weights are the first thing waited for; streamed ones are behind the window's pieces
        ("sparq_conv_window_kernel", 1): [("bar_b_full", "true"), ("bar_win_full", "true"), ("bar_win_xf", "true"), ("bar_b_full", None),
                                          ("ops_bar", streamed), ("ops_bar", streamed), ("bar_b_full", None), ("bar_b_full", None),
                                          ("bar_win_xf", streamed), ("bar_win_full", streamed)],
        ("sparq_conv_window_kernel", 3): [("bar_win_full", "true")]}


def test_no_access_before_the_wait():
    seen = []
    for f, name, body in kernels():
        before = without_lambdas(body[:body.index("dep_wait();")])
        hit = READS.search(before)
        assert not hit, f"{f}: {name} calls {hit.group(0)} before dep_wait()"
        assert not re.search(r"if \([^)]*\)\s*$", before), f"{f}: {name} waits only sometimes"
        seen.append(name)
    assert len(seen) >= 11, seen


@pytest.mark.gpu
@pytest.mark.parametrize("c,hw,r", [(128, 28, 3), (512, 7, 1), (48, 35, 5)])
def test_weights_written_by_the_operation_before(c, hw, r):
    """Weights that a copy, or the library's own 2:4 expansion, has just written."""
    import paper_2105_11010_b200 as sparq
    x = synth.activations(c, (1, hw, hw, c), 0.5)
    p = sparq.SparqParams()
    xd = torch.from_numpy(x).cuda()
    ws = [synth.weights(i, (64, r, r, c)) for i in (1, 2)]
    want = [oracle.conv2d_nhwc(x, w, (1, 1), (r // 2, r // 2), p.mode, 4, 0x1F, 1) for w in ws]
    wd, cur = [torch.from_numpy(w).cuda() for w in ws], torch.empty((64, r, r, c), dtype=torch.int8, device="cuda")
    acc = [torch.empty((1, hw, hw, 64), dtype=torch.int32, device="cuda") for _ in range(20)]
    for i, a in enumerate(acc):
        cur.copy_(wd[i & 1])
        sparq.sparq_conv2d_nhwc_s8(xd, cur, (1, 1), (r // 2, r // 2), p, acc_out=a)
    sparq.sparq_check()
    for i, a in enumerate(acc):
        assert np.array_equal(a.cpu().numpy(), want[i & 1])
    A, b = synth.activations(3, (64, 256), 0.5), sparq.SparqParams(sparq.MODE_BSPARQ)
    sparse = [synth.sparse24_weights(i, 64, 256) for i in (1, 2)]
    dev = [tuple(torch.from_numpy(t).cuda() for t in s) for s in sparse]
    Ad, w = torch.from_numpy(A).cuda(), torch.empty((64, 256), dtype=torch.int8, device="cuda")
    acc = [torch.empty((64, 64), dtype=torch.int32, device="cuda") for _ in range(20)]
    for i, a in enumerate(acc):
        sparq.sparq_sparse24_expand_weights(*dev[i & 1], b, w)
        sparq.sparq_gemm_s8_sparse24(Ad, w, b, acc_out=a)
    sparq.sparq_check()
    for i, a in enumerate(acc):
        assert np.array_equal(a.cpu().numpy(), oracle.gemm_sparse24(A, *sparse[i & 1], b.mode, 4, 0x1F, 1))
