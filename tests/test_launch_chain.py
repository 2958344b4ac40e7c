"""Kernels launched to overlap the one before them (launch_pdl) read memory that
the earlier kernel is still writing when they become resident.  Checked on the
sources: such a kernel waits first (pdl_begin as its first statement), none of
its pointers is __restrict__ (its loads could be taken for loads of constant
memory and moved over the wait), and every kernel launched so is one of them."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_1907_02814_gb300" / "csrc"


def kernels():
    """name -> (parameter list, body's first statement)"""
    found = {}
    for path in sorted(CSRC.glob("*.cu*")):
        text = re.sub(r"//[^\n]*", "", path.read_text())
        for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\((?:[^()]|\([^()]*\))*\)\s*)?(\w+)\s*\(", text):
            depth, i = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(text[i], 0)
                i += 1
            if text[i:].lstrip().startswith("{"):
                found[m.group(1)] = (text[m.end():i - 1], text[i:].lstrip()[1:].lstrip().split(";")[0].strip())
    return found


def test_overlapped_kernels_wait_first_and_take_no_restrict_pointers():
    ks = kernels()
    launched = set()
    for path in sorted(CSRC.glob("*.cu")):
        launched |= set(re.findall(r"launch_pdl\((\w+_kernel)", path.read_text()))
    assert len(launched) >= 8 and launched <= set(ks)
    waiting = {n for n, (_, first) in ks.items() if first == "pdl_begin()"}
    assert launched == waiting
    for name in sorted(launched):
        assert "__restrict__" not in ks[name][0], name
