"""What a rebuild looks at: every file that a source includes from the tree is a
dependency of every object, whatever its suffix.  Objects built before and
after a change of a shared structure must not be linked together."""
import os
import re

from paper_1707_00516_gb300 import build


def test_every_included_file_is_a_dependency():
    deps = {os.path.realpath(p) for p in build._deps()}
    assert os.path.realpath(os.path.join(build.CSRC, "internal.h")) in deps
    for src in sorted(deps):
        if not src.endswith((".cu", ".cuh", ".h")):
            continue
        for name in re.findall(r'#include "([^"]+)"', open(src).read()):
            found = [p for d in (build.CSRC, build.INCLUDE) if os.path.exists(p := os.path.join(d, name))]
            assert found, (src, name)
            assert os.path.realpath(found[0]) in deps, (src, name)
