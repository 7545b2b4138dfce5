"""Kernels that may start while their predecessor drains wait before they touch its results, and that only orders loads which the
compiler may not move: a read-only load (__ldg) or a pointer that is __restrict__ promises that nobody else writes the
memory while the kernel runs, so neither is allowed on anything that earlier work of the stream writes.  The rotation is
uploaded before any kernel.  (No run can show the order; the sources can.)"""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2605_02905_b200" / "csrc"
CONSTANT = {"pi", "pi_t"}   # the rotation


def _code(path):
    return re.sub(r"//[^\n]*", "", path.read_text())


def _arguments(text, start):
    """The text between the parenthesis at or after `start` and its partner."""
    a = text.index("(", start)
    depth = 0
    for i in range(a, len(text)):
        depth += (text[i] == "(") - (text[i] == ")")
        if depth == 0:
            return text[a + 1:i]
    raise AssertionError("unbalanced parentheses")


@pytest.mark.parametrize("path", sorted(CSRC.glob("*.cu*")), ids=lambda p: p.name)
def test_nothing_that_earlier_kernels_write_is_read_as_constant(path):
    text = _code(path)
    for m in re.finditer(r"__ldg\b", text):
        assert CONSTANT & set(re.findall(r"\w+", _arguments(text, m.end()))), _arguments(text, m.end())
    for m in re.finditer(r"\w+_kernel(?=\()", text):
        head = text[max(0, text.rfind("}", 0, m.start())):m.start()]
        if "__global__" not in head or "pdl_wait()" not in text:
            continue
        for p in re.findall(r"__restrict__\s+(\w+)", _arguments(text, m.end())):
            assert p in CONSTANT, (m.group(), p)


def test_the_kernels_are_found():
    """The check above looks at every dependent kernel: each is declared in a file that waits."""
    found = [m for p in CSRC.glob("*.cu") if "pdl_wait()" in _code(p) for m in re.findall(r"(\w+_kernel)(?=\()", _code(p))]
    assert len(set(found)) >= 10, found
