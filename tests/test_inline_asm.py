"""Inline assembly that touches memory is ordered by the compiler: `volatile` (neither merged nor moved across other
volatile statements, such as the wait for the previous kernel) and a "memory" clobber (not moved across stores)."""
from __future__ import annotations

import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_20403_gb300", "csrc")


def statements(text):
    """(volatile?, body) of every asm statement, the body up to the parenthesis that closes it."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"\basm\s*(volatile)?\s*\(", text):
        depth, i, quoted = 1, m.end(), False
        while depth:
            c = text[i]
            if c == '"':
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
            i += 1
        yield bool(m.group(1)), text[m.end():i - 1]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_memory_access_is_ordered(path):
    for volatile, body in statements(open(path).read()):
        if re.search(r"\b(ld|st|red|atom|cp|fence|griddepcontrol|barrier)\.", body):
            assert volatile and re.search(r':\s*"memory"\s*$', body.strip()), body
