"""A bounded wait ends per thread, and what follows it in the tensor-core kernels is the whole warp's or group's work (`.aligned`
tensor-memory instructions, barriers): lanes must not part over its outcome.  So a wait is one lane's, or the whole warp's
(mbar_wait_warp, a vote), or its outcome goes through the group's next barrier with nothing decided by it before.  (No run can show
what happens when a wait gives up half-way through a warp; the sources can.)"""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2605_02905_b200" / "csrc"
KERNELS = [p for p in sorted(CSRC.glob("*.cu")) if "mbar_wait" in p.read_text() and p.name != "eosq_selftest.cu"]


def _headers(code, pos):
    """The statement heads of the blocks around `pos`, innermost first, and the text of the innermost one."""
    heads, depth, inner = [], 0, None
    for i in range(pos, -1, -1):
        if code[i] == "}":
            depth += 1
        elif code[i] == "{":
            if depth:
                depth -= 1
            else:
                heads.append(code[max(code.rfind(c, 0, i) for c in ";{}") + 1:i])
                inner = i if inner is None else inner
    depth = 0
    for j in range(inner, len(code)):
        depth += (code[j] == "{") - (code[j] == "}")
        if depth == 0:
            break
    return heads, code[inner:j]


@pytest.mark.parametrize("path", KERNELS, ids=lambda p: p.name)
def test_lanes_stay_together_after_a_wait(path):
    code = re.sub(r"//[^\n]*", "", path.read_text())
    waits = list(re.finditer(r"\bmbar_wait\(", code))
    assert waits or "mbar_wait_warp(" in code
    for m in waits:
        heads, block = _headers(code, m.start())
        statement = code[max(code.rfind(c, 0, m.start()) for c in ";{}") + 1:code.index(";", m.start())]
        if "&scratch" in statement:
            continue   # the clean-up, which ignores the outcome
        if any(re.search(r"if \((lane|tid) == 0\b", h) for h in heads):
            continue
        kept = re.match(r"\s*const bool (\w+) =", statement)
        assert kept, statement
        name = kept.group(1)
        assert re.search(r"_any\((\w+, )?!%s\)" % name, block), statement
        assert not re.search(r"if \(!?%s\b" % name, block), statement


def test_the_kernels_are_found():
    assert {p.name for p in KERNELS} >= {"eosq_tc.cu", "eosq_quant_ws.cu", "eosq_decode_tc.cu", "eosq_scores_ws.cu"}
