"""Order of memory between the two kernels of the backward tail that run beside one another, as the source has it: a launch that is released early
promises nothing about memory, so the results of the gradient stages are handed over by a release and an acquire."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_08874_b200", "csrc")


def body(src, kernel):
    start = src.index(f" {kernel}(const TailArgs a) {{")
    return src[start:src.index("\n}\n", start)]


def test_conv_tail_hands_over_between_its_wait_and_its_release():
    src = open(os.path.join(CSRC, "bwd_tail.cu")).read()
    conv = body(src, "bwd_conv_tail_kernel")
    assert 0 < conv.index("pdl_wait_prior();") < conv.index("store_release(a.handed") < conv.index("pdl_release_next();")
    assert re.search(r"void store_release\(.*st\.release\.gpu", src) and "ld.acquire.gpu" in src


def test_pool_tail_takes_over_before_it_reads():
    src = open(os.path.join(CSRC, "bwd_tail.cu")).read()
    pool = body(src, "bwd_pool_tail_kernel")
    beside = pool[pool.index("__syncthreads_or("):]
    # a block that does not see the word waits for the kernel before; nothing of the stages is read earlier
    assert re.match(r"__syncthreads_or\(threadIdx\.x == 0 && load_acquire\(a\.handed\)\)\) \{\s*pdl_wait_prior\(\);", beside)
    for read in ("a.da", "a.dq"):
        assert read not in pool[:pool.index("__syncthreads_or(")]
    # what comes next in the stream waits for this kernel alone: it ends after the kernel before
    assert re.search(r"if \(BESIDE\) \{\s*pdl_release_next\(\);\s*pdl_wait_prior\(\);\s*\}\s*$", pool)
