"""The waits of the direct kernels' pipeline, checked in the source: a missing reconvergence is undefined
behaviour on the GPU and shows there only by chance."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_06007_gb300", "csrc")


def _body(src, name):
    """The text of the function whose definition `name(` starts, braces matched."""
    at = src.index("{", src.index(name + "("))
    depth = 0
    for i in range(at, len(src)):
        depth += {"{": 1, "}": -1}.get(src[i], 0)
        if depth == 0:
            return src[at:i + 1]
    raise AssertionError(name)


def test_warps_meet_before_aligned_instructions():
    # tcgen05.ld and tcgen05.wait::ld are .aligned: every wait of the warps that use them is a whole
    # warp's, and only the issuing thread waits by itself.
    src = open(os.path.join(CSRC, "k_direct.cu")).read()
    item = _body(src, " direct_item")
    assert "tmem_load_wait" in item and len(re.findall(r"\bwarp_wait\(", item)) >= 3
    assert not re.search(r"\bpipe_wait\(|\bmbar_wait\(", item), "a per-thread wait in front of aligned instructions"
    assert re.search(r"pipe_wait\(.*?\);\s*__syncwarp\(\);\s*}$", _body(src, "void warp_wait"), re.S)


def test_products_end_before_tensor_memory_is_freed():
    # A wait that ran out stops the issuing thread, and what it had issued is waited for (with a
    # limit) before the CTA gives its memory back.
    src = open(os.path.join(CSRC, "k_direct.cu")).read()
    issue, end = _body(src, "void issue_chunks"), _body(src, "void direct_end")
    assert len(re.findall(r"\bok = [^;]*pipe_wait\([^;]*;", issue)) == len(re.findall(r"pipe_wait\(", issue)) == 2
    assert issue.rindex("pipe_wait(") < issue.index("if (!ok) break;") < issue.index("tc::mma<")
    assert end.index("mma_commit(&sh.drained)") < end.index("mbar_try(&sh.drained") < end.index("tmem_free")
