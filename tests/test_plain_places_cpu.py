"""Plain launches that do not fill the GPU start after the query preparation,
not beside it: beside it their CTAs go where its blocks are not, two to an SM,
while other SMs stay idle.  Which launches those are, and that the launch asks.
Host arithmetic and source only."""
import os
import re

import pytest

from host import ctx_hooks
from paper_1707_00516_gb300 import build


@pytest.mark.parametrize("n_q,n_refs,fills", [(1000, 1000, 0), (1000, 4600, 0), (1000, 5000, 1), (1, 300, 0), (128, 38_800, 1),
                                              (128, 38_600, 0)])
def test_fills(tmp_path, n_q, n_refs, fills):
    # two CTAs on each of 152 SMs; 128 references a unit, of databases padded to 256
    assert ctx_hooks(tmp_path).hook_plain_fills(304, 128, n_q, n_refs) == fills


def test_launch_asks():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, "plain.cu")).read())
    launches = [ln.strip() for ln in src.split("\n") if "launch_dependent(" in ln]
    assert launches == ["if (part.fills) return launch_dependent(fn, dim3((unsigned)part.grid), dim3(PL_THREADS), smem, s, a);"]
