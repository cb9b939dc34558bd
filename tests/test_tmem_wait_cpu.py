"""Loads from TMEM, read from the source: the registers that a tcgen05.ld names
hold its values only after tcgen05.wait::ld, so the wait has to be in the same
asm block, or name the registers as its own operands; a wait that only clobbers
memory lets the compiler use them before it.  Nothing here runs on a GPU."""
import glob
import os
import re

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_00516_gb300")


def asm_blocks():
    """(file, asm statement) in order of the source."""
    for path in sorted(glob.glob(os.path.join(PKG, "csrc", "*.cu*")) + glob.glob(os.path.join(PKG, "probe", "*.cu"))):
        src = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"asm volatile\(", src):
            end, depth = m.end(), 1
            while depth:
                depth += {"(": 1, ")": -1}.get(src[end], 0)
                end += 1
            yield os.path.basename(path), src[m.start():end]


def registers(block):
    return set(re.findall(r'"[=+]r"\((v\[\d+\])\)', block))


def test_every_load_is_tied_to_its_wait():
    blocks = list(asm_blocks())
    loads = [i for i, (_, b) in enumerate(blocks) if "tcgen05.ld." in b]
    assert len(loads) >= 4
    for i in loads:
        path, body = blocks[i]
        assert registers(body), (path, body)
        if "tcgen05.wait::ld" not in body:
            after_path, after = blocks[i + 1]
            assert after_path == path and "tcgen05.wait::ld" in after, (path, body)
            assert registers(body) <= registers(after), (path, body, after)
