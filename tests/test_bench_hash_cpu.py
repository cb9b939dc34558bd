"""The source hash that bench.py's recorded DRAM figures are keyed by covers every
file of the kernel: its source and each header that this includes, directly or
through another."""
import os
import re

import pytest

import bench
from paper_1707_00516_gb300 import build


def included(name, seen):
    if name in seen or not os.path.exists(os.path.join(build.CSRC, name)):
        return seen  # (the public header declares no kernel code)
    seen.add(name)
    for nxt in re.findall(r'#include "([^"]+)"', open(os.path.join(build.CSRC, name)).read()):
        included(nxt, seen)
    return seen


@pytest.mark.parametrize("form,source", [("fp4", "tensor.cu"), ("plain", "plain.cu")])
def test_hash_covers_the_kernels_files(monkeypatch, form, source):
    read = []
    real = open

    def spy(path, *a, **kw):
        read.append(os.path.basename(str(path)))
        return real(path, *a, **kw)

    files = included(source, set())
    monkeypatch.setattr("builtins.open", spy)
    bench.kernel_source_hash(form)
    monkeypatch.undo()
    assert set(read) == files
