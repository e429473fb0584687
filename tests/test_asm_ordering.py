"""Inline PTX that orders memory says so to the compiler.

A wait, fence, commit, tensor-core or tensor-memory instruction without a
"memory" clobber lets the compiler move plain shared-memory loads and stores
across it (a record read before the wait for its copy, a tile stored after the
fence that publishes it).  Every asm statement of the kernel sources with such an
instruction is volatile and clobbers "memory", and a tcgen05.ld stands in one
statement with its wait, before which its registers hold nothing.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_15511_gb300", "csrc")
ORDERING = re.compile(r"mbarrier|fence|tcgen05|cp\.async|bar\.sync|barrier")


def asm_statements(text):
    """(volatile, statement) of every asm in the text, comments removed."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"\basm\b(\s+volatile)?\s*\(", text):
        depth, quoted, i = 1, False, m.end()
        while depth:
            ch = text[i]
            if ch == '"' and text[i - 1] != "\\":
                quoted = not quoted
            elif not quoted:
                depth += (ch == "(") - (ch == ")")
            i += 1
        yield bool(m.group(1)), text[m.end():i - 1]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_ordering_statements_clobber_memory(path):
    with open(path) as f:
        for volatile, stmt in asm_statements(f.read()):
            if not ORDERING.search(stmt):
                continue
            assert volatile, stmt
            assert re.search(r':\s*"memory"\s*$', stmt), stmt
            if "tcgen05.ld" in stmt:
                assert "tcgen05.wait::ld" in stmt, stmt


def test_the_scan_finds_the_statements():
    with open(os.path.join(CSRC, "legendre_tc.cu")) as f:
        found = [s for _, s in asm_statements(f.read()) if ORDERING.search(s)]
    for what in ("mbarrier.try_wait", "tcgen05.mma", "tcgen05.ld", "tcgen05.st", "fence.proxy.async", "cp.async.bulk"):
        assert any(what in s for s in found), what
