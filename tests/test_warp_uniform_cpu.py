"""Branches of a whole warp in the few-query kernel, read from its source.

A warp's lanes meet at whole-warp instructions (votes, reductions, elect.sync),
so what decides a branch around one has to be the same in every lane.  A value
that other warps or CTAs change -- a barrier's state, a flag, a shared cut -- is
read by each lane for itself, and two lanes that read differently would wait
for each other without end.  Such a value has to pass through a vote or a
broadcast first.  Nothing here runs on a GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_00516_gb300", "csrc")
VOTE = re.compile(r"__(all|any)_sync\(|__shfl_sync\(")


def kernel(path, name):
    """Source of one kernel, comments out, one statement or block head a line."""
    src = open(os.path.join(CSRC, path)).read()
    src = re.sub(r"//[^\n]*", "", src)
    at = src.index(f" {name}(")
    at = src.index("{", src.index(")", at))
    depth, end = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(src[end], 0)
        end += 1
        if depth == 0:
            break
    return re.sub(r"\s+", " ", src[at:end]).replace("; ", ";\n").replace("{ ", "{\n").replace("} ", "}\n").split("\n")


@pytest.fixture(scope="module")
def few():
    return kernel("few.cu", "few_kernel")


def test_waits_of_a_whole_warp_are_entered_by_a_vote(few):
    """A branch around warp_wait tests nothing but a vote."""
    waits = [i for i, ln in enumerate(few) if "warp_wait(" in ln]
    assert len(waits) >= 6
    for i in waits:
        if few[i - 1].startswith("if (") and few[i - 1].endswith("{"):
            assert VOTE.search(few[i - 1]), few[i - 1]


@pytest.mark.parametrize("value,read", [("ended", "finished"), ("now", "load_cut")])
def test_values_of_other_warps_are_made_uniform(few, value, read):
    lines = [ln for ln in few if re.search(rf"\b{value} = ", ln) and read in ln]
    assert lines
    for ln in lines:
        assert VOTE.search(ln), ln


def test_the_abort_flag_is_voted_on(few):
    lines = [ln for ln in few if ln.startswith("if (") and "*abort_flag" in ln]
    assert lines
    for ln in lines:
        assert VOTE.search(ln), ln
