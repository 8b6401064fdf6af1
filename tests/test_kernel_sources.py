"""CPU check of the kernel sources: inline PTX that several lanes execute
together (shuffles, votes, barriers and the like, ".sync") is `asm volatile`.
Without it the compiler may delete, duplicate or move the statement, for
instance under a branch that only some of the lanes take, where the others
named in its mask never arrive."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2209_08196_gb300", "csrc")
SOURCES = sorted(os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*.cu*")))


def asm_statements(text):
    """(is volatile, the statement up to its closing ");") of every asm."""
    for m in re.finditer(r"\basm\b(\s+volatile\b)?\s*\(", text):
        yield m.group(1) is not None, text[m.start():text.index(");", m.end()) + 2]


@pytest.mark.parametrize("name", SOURCES)
def test_warp_wide_asm_is_volatile(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    loose = [a for volatile, a in asm_statements(text) if ".sync" in a and not volatile]
    assert not loose, loose


def test_the_sources_have_such_statements():
    found = 0
    for name in SOURCES:
        with open(os.path.join(CSRC, name)) as f:
            found += sum(".sync" in a for _, a in asm_statements(f.read()))
    assert found >= 1
