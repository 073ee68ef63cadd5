"""The kernels with warp roles wait for the kernel before in each role by itself: every branch that reads or writes the
caller's memory waits before it does, on every path.  (tests/test_dependency_wait.py looks at the text up to a kernel's first
wait, which in these is the producer's.)"""
import os
import re

import numpy as np
import pytest
import torch

import oracle
import sparq_synth as synth
from test_dependency_wait import CSRC, READS, block_end, kernel_bodies, roles

WAIT = re.compile(r"\bdep_wait\(\);")


def device_functions():
    """name -> body of the functions that kernels call, all headers together."""
    out = {}
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
            for m in re.finditer(r"__device__[^;{}()]*?(\w+)\s*\(", text):
                depth, j = 1, m.end()
                while depth:
                    depth += {"(": 1, ")": -1}.get(text[j], 0)
                    j += 1
                a = re.match(r"\s*\{", text[j:])
                if a:
                    out[m.group(1)] = out.get(m.group(1), "") + text[j:block_end(text, j + a.end() - 1)]
    return out


def touching_functions():
    """Functions that read or write global memory, by themselves or through another one."""
    bodies = device_functions()
    own = re.compile(r"\.global\b|__ldg|__ldcs|__stcs|cp\.async\.bulk\.tensor|\b(?:u8_out|f32_out|acc_out|residual)\s*\[|reinterpret_cast<[^>]*\*>\((?:out|e\.\w+)\b")
    # prefetch_tensormap: a kernel argument; mbar_wait: the library's status word
    known = {n for n, b in bodies.items() if own.search(b)} - {"prefetch_tensormap", "mbar_wait", "dep_wait"}
    while True:
        more = {n for n, b in bodies.items() if n not in known and any(re.search(r"\b%s\s*(?:<[^;(]*>)?\(" % k, b) for k in known)}
        if not more:
            return known
        known |= more


def strip_lambdas(text, touching):
    """(text without the bodies of named lambdas, names of those whose bodies touch memory)."""
    names, out, i = set(), "", 0
    for m in re.finditer(r"auto (\w+) = \[&\][^;{]*\{", text):
        if m.start() < i:
            continue
        end = block_end(text, m.end() - 1)
        if touching(text[m.end():end], names):
            names.add(m.group(1))
        out += text[i:m.start()]
        i = end
    return out + text[i:], names


def blocks_around(text, at):
    """Start positions of the blocks that enclose position `at`, outermost first."""
    open_ = []
    for j in range(at):
        if text[j] == "{":
            open_.append(j)
        elif text[j] == "}" and open_:
            open_.pop()
    return open_


def unguarded(setup, role, functions):
    """The first access of a role's branch that no wait comes before on every path, and its number of accesses."""
    call = re.compile(r"\b(%s)\s*(?:<[^;(]*>)?\(" % "|".join(sorted(functions)))

    def first(text, names):
        hits = [m for m in READS.finditer(text) if not m.group(1).startswith("issue_")] + list(call.finditer(text))      # issue_*: lambdas
        hits += [m for n in names for m in re.finditer(r"\b%s\(" % n, text)]
        return sorted(hits, key=lambda m: m.start())

    _, outer = strip_lambdas(setup, first)
    text, names = strip_lambdas(role, lambda t, n: first(t, n | outer))
    waits = [m.start() for m in WAIT.finditer(text) if re.search(r"[;{}]\s*$", text[:m.start()])]      # not `if (x) dep_wait();`
    around = [blocks_around(text, w) for w in waits]
    hits = first(text, names | outer)
    for h in hits:
        here = blocks_around(text, h.start())
        if not any(w < h.start() and here[:len(b)] == b for w, b in zip(waits, around)):
            return h.group(0), len(hits)
    return None, len(hits)


def role_kernels():
    return [(f, name, *roles(body)) for f, name, body in kernel_bodies() if roles(body)[1]]


def test_functions_that_touch_memory_are_found():
    known = touching_functions()
    assert {"tma_load_2d", "tma_load_row_groups", "tma_load_im2col_4d", "tma_load_4d", "tma_store_2d", "epi_stage_scale_bias", "epi_frag_columns",
            "epi_general", "epi_warp_columns"} <= known, known
    assert not known & {"mbar_try_wait", "xform_fused", "tmem_ld_wait", "tc_mma_i8_if", "make_epi_view", "elect_one"}, known


def test_every_role_waits_before_its_first_access():
    functions, found = touching_functions(), {}
    for f, name, setup, branches in role_kernels():
        text, names = strip_lambdas(setup, lambda t, n: None)
        assert not READS.search(text) and not WAIT.search(text), name
        for i, role in enumerate(branches):
            hit, accesses = unguarded(setup, role, functions)
            assert hit is None, f"{f}: {name}, role {i}: {hit} before dep_wait()"
            if accesses:
                found.setdefault(name, set()).add(i)
    # producer and epilogue; the small form's MMA warp also fetches the first weights
    assert found == {"sparq_gemm_kernel": {0, 2}, "sparq_conv_window_kernel": {0, 2}, "sparq_gemm_sparse24_kernel": {0, 2},
                     "sparq_gemm_small_kernel": {0, 1, 2}}, found


def test_each_of_these_waits_is_missed():
    """The check sees every one of the waits: without it, or with a condition in front of it, an access is unguarded."""
    functions, waits = touching_functions(), 0
    for f, name, setup, branches in role_kernels():
        for role in branches:
            if unguarded(setup, role, functions)[1]:
                for m in WAIT.finditer(role):
                    waits += 1
                    for instead in ("", "if (lane == 0) dep_wait();", "if (lane == 0) { dep_wait(); }"):
                        assert unguarded(setup, role[:m.start()] + instead + role[m.end():], functions)[0], (name, role[m.start() - 200:m.end()])
    assert waits == 9


@pytest.mark.gpu
@pytest.mark.parametrize("nb,hw,c,cout,r,stride", [
    (1, 14, 256, 64, 1, 1),       # small form
    (24, 28, 64, 256, 1, 1),      # full form, several column tiles
    (25, 39, 64, 256, 1, 2),      # the same through an im2col map
    (8, 28, 128, 128, 3, 1)])     # windows
def test_epilogue_operands_written_by_the_operation_before(nb, hw, c, cout, r, stride):
    """Scale, bias and residual that a copy, or a kernel of this library, has just written, and an output that the kernel
    before still reads."""
    import paper_2105_11010_b200 as sparq
    p, none, pad = sparq.SparqParams(), sparq.SparqParams(sparq.MODE_NONE), r // 2
    x, w = synth.activations(c, (nb, hw, hw, c), 0.5), synth.weights(c, (cout, r, r, c))
    ho = (hw + 2 * pad - r) // stride + 1
    inv, sets = synth.inv_out_scale(r * r * c), []
    for i in range(2):
        sets.append((synth.scales(i, cout), synth.bias(i + 5, cout), synth.activations(i + 9, (nb, ho, ho, cout), 0.5)))
    acc = oracle.conv2d_nhwc(x, w, (stride, stride), (pad, pad), p.mode, 4, 0x1F, 1)
    want = [oracle.epilogue(acc, s, b, True, inv, residual=q, residual_scale=0.5)[1] for s, b, q in sets]
    assert not np.array_equal(*want)
    xd, wd = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
    dev = [[torch.from_numpy(t).cuda() for t in s] for s in sets]
    scale, bias, res = [torch.empty_like(t) for t in dev[0]]
    out = torch.empty_like(res)
    kept = [torch.empty_like(out) for _ in range(20)]
    for i, k in enumerate(kept):
        s, b, q = dev[i & 1]
        scale.copy_(s)
        bias.copy_(b)
        sparq.sparq_quantize(q, res, nb * ho * ho, cout, none)
        sparq.sparq_conv2d_nhwc_s8(xd, wd, (stride, stride), (pad, pad), p, scale=scale, bias=bias, relu=True, inv_out_scale=inv,
                                   u8_out=out, residual=res, residual_scale=0.5)
        sparq.sparq_quantize(out, k, nb * ho * ho, cout, none)
    sparq.sparq_check()
    for i, k in enumerate(kept):
        assert np.array_equal(k.cpu().numpy().reshape(want[0].shape), want[i & 1]), i


@pytest.mark.gpu
def test_scale_and_bias_of_the_24_product_written_by_the_operation_before():
    import paper_2105_11010_b200 as sparq
    m, k, n = 148 * 256 + 77, 256, 128
    p, none = sparq.SparqParams(), sparq.SparqParams(sparq.MODE_NONE)
    A, sparse = synth.activations(3, (m, k), 0.5), synth.sparse24_weights(1, n, k)
    inv, sets = synth.inv_out_scale(k // 2), [(synth.scales(i, n), synth.bias(i + 5, n)) for i in range(2)]
    acc = oracle.gemm_sparse24(A, *sparse, p.mode, 4, 0x1F, 1)
    want = [oracle.epilogue(acc, s, b, True, inv)[1] for s, b in sets]
    assert not np.array_equal(*want)
    w = torch.empty((n, sparq.sparq_sparse24_expanded_k(k, p)), dtype=torch.int8, device="cuda")
    sparq.sparq_sparse24_expand_weights(*[torch.from_numpy(t).cuda() for t in sparse], p, w)
    Ad, dev = torch.from_numpy(A).cuda(), [[torch.from_numpy(t).cuda() for t in s] for s in sets]
    scale, bias = [torch.empty_like(t) for t in dev[0]]
    out, work = torch.empty((m, n), dtype=torch.uint8, device="cuda"), torch.empty((m, 3 * k), dtype=torch.uint8, device="cuda")
    kept = [torch.empty_like(out) for _ in range(20)]
    for i, q in enumerate(kept):
        scale.copy_(dev[i & 1][0])
        bias.copy_(dev[i & 1][1])
        sparq.sparq_gemm_s8_sparse24(Ad, w, p, workspace=work, scale=scale, bias=bias, relu=True, inv_out_scale=inv, u8_out=out)
        sparq.sparq_quantize(out, q, m, n, none)
    sparq.sparq_check()
    for i, q in enumerate(kept):
        assert np.array_equal(q.cpu().numpy(), want[i & 1]), i
