"""No CTA of a cluster may leave while a peer can still write to its shared memory.

The give-up path of the cluster form cannot be run on purpose (a CTA that has left while its peers
still store to it is a memory fault), so the order of its steps is checked in the source: a CTA
that gave up a wait stays, after its own last remote store, until the rest of the cluster has sent
everything and until those bytes have landed.
"""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2105_11010_b200", "csrc")


def kernel_source():
    text = open(os.path.join(CSRC, "sparq_gemm_small_kernel.cuh")).read()
    text = re.sub(r"//[^\n]*", "", text)
    start = text.index("sparq_gemm_small_kernel(const")
    return text[start:text.index("cudaError_t launch_gemm_small(", start)]


def test_a_cta_that_gave_up_stays_for_its_senders():
    src = kernel_source()
    last_store = src.rindex("store_remote16(")
    leave = src.index("tcgen05.dealloc")
    stay = re.search(r"if \(SHARED && split > 1 && \*abort_flag\) \{(.*?)\n    \}", src, re.S)
    assert stay and last_store < stay.start() < leave
    # every thread of the CTA takes the same side: the flag is read behind a barrier of the whole CTA
    assert re.search(r"__syncthreads\(\);\s*$", src[:stay.start()])
    body = stay.group(1)
    assert body.index("cluster_arrive();") < body.index("cluster_wait();") < body.index("mbar_wait(smem_u32(&bar_recv), 0")
    assert body.rstrip().endswith("true);")        # not cut short by the flag itself


def test_remote_stores_do_not_depend_on_the_abort_flag():
    src = kernel_source()
    sender = src[src.rindex("cluster_wait();", 0, src.rindex("store_remote16(")):src.rindex("store_remote16(")]
    assert "abort_flag" not in sender and "return" not in sender


def test_aligned_barriers_follow_a_converged_warp():
    src = kernel_source()
    assert all(re.search(r"__syncwarp\(\);\s*$", src[:m.start()]) for m in re.finditer(r"cluster_arrive\(\);", src))
