"""Inline PTX that all lanes or threads must reach together is volatile (no GPU).

An asm statement without `volatile` may be moved to where its result is used.  For an instruction that
names the lanes taking part (`redux.sync`), or that waits or orders memory, a use inside a divergent
branch would then let it run with lanes missing: the result is undefined and the warp may hang.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01654_gb300", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h")))
TOGETHER = re.compile(r"\.sync\b|\bbar(rier)?\.|mbarrier|griddepcontrol|\bfence\b|cp\.(async|reduce)|membar|tcgen05")


def asm_statements(text):
    """(qualifiers, template) of every asm statement."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)
    for m in re.finditer(r"\basm\b\s*((?:volatile|__volatile__)?)\s*\(((?:\s*\"(?:[^\"\\]|\\.)*\")+)", text):
        yield m.group(1), m.group(2)


@pytest.mark.parametrize("path", SOURCES, ids=[os.path.basename(p) for p in SOURCES])
def test_collective_instructions_are_volatile(path):
    movable = [t.strip() for q, t in asm_statements(open(path).read()) if TOGETHER.search(t) and not q]
    assert not movable, f"asm without volatile: {movable}"


def test_the_statements_are_found():
    found = [t for p in SOURCES for _, t in asm_statements(open(p).read()) if TOGETHER.search(t)]
    assert any("redux.sync" in t for t in found) and any("griddepcontrol" in t for t in found)
