"""Inline assembly that orders memory must say so to the compiler.  `volatile` keeps such a statement in line with other
volatile statements only; ordinary loads and stores may cross it unless it clobbers "memory".  Read from the sources, since
a reordering would be a race on the GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_01334_gb300", "csrc")
# barriers, fences, asynchronous copies and their waits, tensor-core issue, commit and tensor memory
ORDERING = re.compile(r"mbarrier\.|fence|cp\.async|tcgen05\.|bar\.sync|membar")


def statements():
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh", ".h")):
            continue
        s = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"\basm\s*(volatile\s*)?\(", s):
            depth, i, instr = 1, m.end(), False
            while depth:  # to the closing parenthesis, strings skipped
                c = s[i]
                if c == '"' and s[i - 1] != "\\":
                    instr = not instr
                depth += 0 if instr else (c == "(") - (c == ")")
                i += 1
            yield f, s.count("\n", 0, m.start()) + 1, bool(m.group(1)), s[m.end():i - 1]


FOUND = [x for x in statements() if ORDERING.search(x[3])]


def test_statements_are_found():
    assert len(FOUND) >= 20, len(FOUND)


@pytest.mark.parametrize("f,line,volatile,text", FOUND, ids=["%s:%d" % x[:2] for x in FOUND])
def test_ordering_statement_clobbers_memory(f, line, volatile, text):
    assert volatile, text
    assert re.search(r':[^:"]*"memory"', text), text


def test_tensor_memory_load_waits_in_its_own_statement():
    """The registers of tcgen05.ld are not valid before the wait, and arithmetic on them depends on the load's statement alone."""
    loads = [t for _, _, _, t in FOUND if "tcgen05.ld" in t]
    assert loads
    for t in loads:
        assert "tcgen05.wait::ld" in t.split("tcgen05.ld", 1)[1], t
