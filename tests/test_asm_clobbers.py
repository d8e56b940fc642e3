"""Inline assembly that writes memory (or orders accesses to it) says so: an
asm statement with a store, an asynchronous copy, a reduction, an atomic or a
wait names "memory" among its clobbers, so the compiler keeps ordinary loads
of what it wrote behind it."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_05581_gb300", "csrc")
WRITES = re.compile(r"(?<![\w.])(st|red|atom|cp|mbarrier|fence|membar|bar|barrier)\.")


def _statements(text):
    for m in re.finditer(r"\basm\b(?:\s+volatile)?\s*\(", text):
        depth, i, quoted = 1, m.end(), False
        while depth:
            c = text[i]
            if c == '"' and text[i - 1] != "\\":
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
            i += 1
        yield text.count("\n", 0, m.start()) + 1, text[m.end():i - 1]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_memory_clobber(path):
    with open(path) as f:
        text = f.read()
    bad = [line for line, body in _statements(text) if WRITES.search(body) and '"memory"' not in body]
    assert not bad, f"asm without a memory clobber at line(s) {bad}"
