"""Full barriers of the ring that the two transform teams of sparq_gemm_kernel read in turn.

A parity answers for every second phase of a barrier, so a team may ask for a phase only once it knows that the one
before has completed.  In a ring of an odd number of stages the stage was the other team's before, which nothing
orders before the question: the phase two before would answer, and the team would work on a stage that the other
one still has, or that has not landed.  That is a race on shared memory, so it is looked for in the source and in a
model of the ring; the GPU test runs the odd rings."""
import os
import re

import numpy as np
import pytest
import torch

import oracle
import sparq_synth as synth

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_11010_b200", "csrc")


def kernel_source():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "sparq_gemm_kernel.cuh")).read())
    return text[text.index("sparq_gemm_kernel(const __grid_constant__"):text.index("tcgen05.dealloc.cta_group::1.sync.aligned.b32")]


def test_teams_ask_two_sets_of_full_barriers():
    src = kernel_source()
    role = src[src.index("const XformDev xf = g.xf;"):]
    # which rings have two sets: the one that the teams read, with A in tensor memory and without
    assert "kFullSets = MODE != SPARQ_MODE_NONE && !ATM ? 2 : 1, kRawSets = ATM ? 2 : 1;" in src
    for ring, sets, stages in (("bar_full", "kFullSets", "S"), ("bar_raw", "kRawSets", "SA")):
        assert re.search(r"uint64_t[^;]*\b%s\[[^;\]]*%s \* kMaxStages" % (ring, sets), src)
        assert re.search(r"q < %s \* %s; \+\+q\) mbar_init\(smem_u32\(&%s\[q\]\)" % (sets, stages, ring), src)
    # the producer announces round `use` of a stage on set use & 1
    assert "sets = raw ? kRawSets : kFullSets;" in src and "set = sets == 2 ? 8u * (uint32_t)ring : 0u;" in src
    assert "bars_full + 8u * (uint32_t)s + (use & 1u) * set;" in src
    # and the teams ask for it there, nowhere else: every other barrier of both sets in turn
    for ring, sets, stages, q, ph in (("bar_full", "kFullSets", "S", "q", "ph"), ("bar_raw", "kRawSets", "SA", "qa", "pa")):
        asked = re.findall(r"(\w+)(?:<true>)?\(smem_u32\(&%s\[(\w+)\]\), (\w+)" % ring, role)
        assert sorted(asked) == [("mbar_test", q, ph), ("mbar_wait", q, ph)] and len(re.findall(r"\b%s\b" % ring, role)) == 2
        assert f"int {q} = team;" in role and f"{q} += kXfTeams;" in role
        assert f"if ({q} >= {sets} * {stages}) {{ {q} -= {sets} * {stages}; {ph} ^= 1u; }}" in role


@pytest.mark.parametrize("sets", [1, 2])
@pytest.mark.parametrize("stages", range(2, 9))
def test_model_of_the_ring(stages, sets):
    """Copies that land in any order, within what the release of stages allows: a team that has seen its own items so
    far asks for its next one.  Two sets of barriers answer for that one; one set does in even rings only."""
    rng = np.random.default_rng(stages)
    wrong = 0
    for _ in range(300):
        # items below `released` have been released, in order, and so loaded up to `released + stages`
        released = int(rng.integers(0, 40))
        landed = set(range(released)) | {i for i in range(released, released + stages) if rng.random() < 0.5}
        barrier = lambda i: i % (stages * sets)
        for item in range(released, released + stages):
            if set(range(item % 2, item + 1, 2)) <= landed:
                nxt = item + 2
                done = sum(1 for i in landed if barrier(i) == barrier(nxt))
                says = done % 2 != nxt // (stages * sets) % 2        # the phase under way is not the one asked for
                wrong += says != (nxt in landed)
    assert (wrong > 0) == (sets == 1 and stages % 2 == 1)


@pytest.mark.gpu
@pytest.mark.parametrize("m,k,n,residual,mode,bits", [
    (148 * 128 * 3 + 17, 128, 512, True, 2, 4), (148 * 128 + 1, 256, 1024, True, 2, 4), (148 * 128 * 2 + 5, 256, 288, True, 1, 3),   # three stages
    (148 * 128 * 9 + 45, 128, 64, True, 2, 4),                                                                                   # seven
    (148 * 128 * 2 + 97, 1024, 256, False, 2, 4), (148 * 128 - 3, 2064, 256, False, 2, 2)])                                      # five raw ones
def test_odd_rings(m, k, n, residual, mode, bits):
    import paper_2105_11010_b200 as sparq
    A, B = synth.activations(k, (m, k), 0.5), synth.weights(n, (k, n))
    scale, bias, inv = synth.scales(n, n), synth.bias(n, n), synth.inv_out_scale(k)
    res = synth.activations(n + 1, (m, n), 0.5) if residual else None
    mask = (1 << (9 - bits)) - 1
    dev = [torch.from_numpy(np.ascontiguousarray(t)).cuda() for t in (A, B.T, scale, bias)]
    rd = torch.from_numpy(res).cuda() if residual else None
    out = [torch.empty((m, n), dtype=torch.uint8, device="cuda") for _ in range(20)]
    for o in out:
        sparq.sparq_gemm_s8(dev[0], dev[1], sparq.SparqParams(mode, bits, mask, 1), scale=dev[2], bias=dev[3], relu=True,
                            inv_out_scale=inv, u8_out=o, residual=rd, residual_scale=0.02)
    sparq.sparq_check()
    _, want = oracle.epilogue(oracle.gemm(A, B, mode, bits, mask, 1), scale, bias, True, inv, residual=res, residual_scale=0.02)
    assert np.array_equal(out[0].cpu().numpy(), want)
    assert all(torch.equal(o, out[0]) for o in out[1:])
