"""The tensor kernel's MMA issuer, read from its source: a whole warp runs it and
issues by elect.sync, so its lanes agree on every wait's outcome before they go
on or leave; a wait whose outcome each lane took for itself could leave some at
an elect.sync that the others, whose wait ran out, never reach.  Nothing here
runs on a GPU."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_00516_gb300", "csrc")


def test_issuer_waits_by_vote():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tensor.cu")).read())
    issuer = src[src.index("} else if (warp == 1) {"):src.index("} else if (PK && warp >= 6")]
    assert "mma_stage4" in issuer
    assert issuer.count("warp_wait(") == 3
    assert "mbar_wait(" not in issuer and "mbar_try_wait(" not in issuer
    wait = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tc_ptx.cuh")).read())
    wait = re.search(r"bool warp_wait\([^)]*\) \{(.*?)\n\}", wait, re.S).group(1)
    assert wait.count("__all_sync(0xffffffffu, mbar_") == 2
