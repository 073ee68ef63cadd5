"""Copies in flight when a CTA of the GEMM kernel gives up: none may land after it has left.

Without a transform two producers announce on the same barriers.  They may stop at different stages, and then a stage
that only one of them announced never completes for want of the other's arrival: the one that waits for its copies
would wait out its limit, stage by stage, and leave without knowing.  A wait that runs out cannot be had on demand, so
the order of the steps is checked in the source."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_11010_b200", "csrc")


def kernel_source():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "sparq_gemm_kernel.cuh")).read())
    return text[text.index("sparq_gemm_kernel(const __grid_constant__"):text.index("tcgen05.dealloc.cta_group::1.sync.aligned.b32")]


def test_the_producer_behind_arrives_for_the_other_one():
    src = kernel_source()
    assert "kSharedFull = MODE == SPARQ_MODE_NONE;" in src and "mbar_init(smem_u32(&bar_full[q]), kSharedFull ? 2 : 1);" in src
    assert "announced[0] = announced[1] = kStillIssuing;" in src[:src.index("__syncthreads();")]
    # every producer says where it stopped, aborted or not, before it looks at the flag
    stop = src.index("if (kSharedFull) announced[me] = it;")
    abort = src.index("if (*abort_flag) {", stop)
    assert re.match(r"\s*if \(kSharedFull\) announced\[me\] = it;\s*if \(\*abort_flag\) \{", src[stop:])
    tail = src[abort:]
    arrive = tail.index("for (uint32_t j = it; other != kStillIssuing && j < other; ++j, ++last) mbar_arrive(bars_full")
    assert "j < last; ++j)" in tail[arrive:tail.index("mbar_wait(bars_full")]
    assert tail.index("other = announced[me ^ 1]") < arrive < tail.index("mbar_wait(bars_full")
    assert "clock64() - t0 <= g.wait_limit" in tail[:arrive]             # bounded
    # a stage that did not land is not released: the producers are a ring apart at most
    assert re.search(r"if \(kSharedFull\) \{\s*if \(!mbar_wait<true>\(smem_u32\(&bar_full\[s\]\)[^;]*\) \{ live = false; break; \}", src)
    assert "tile < total_tiles && live;" in src[src.index("make_idesc_i8(BN)"):]
