"""The tensor kernel's epilogue, read from its source: emptying a warp's queues
takes lanes apart (atomics and stores of single lanes), and a whole-warp TMEM
load (tcgen05.ld.sync.aligned) may come next, so it ends with the lanes
together.  Nothing here runs on a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_00516_gb300", "csrc")


def test_flush_ends_with_the_warp_together():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tensor.cu")).read())
    body = re.search(r"auto flush = \[&\]\(\) \{(.*?)\n\s*\};", src, re.S).group(1)
    assert body.split(";")[-2].strip() == "__syncwarp()"
    # nothing between a flush and the load takes the lanes apart again
    loop = src[src.index("> S::QD - G)) flush();"):]
    between = loop[:loop.index("tmem_ld_group")]
    assert "if (" not in between
