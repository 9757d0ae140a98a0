"""No full-mask warp collective stands behind a short-circuit operator: a lane
that the left operand keeps from evaluating it would leave the others waiting for
it (undefined, possibly without end), and be it only where a check fails."""
import glob
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCES = sorted(f for e in ("cu", "cuh", "h") for f in
                 glob.glob(os.path.join(ROOT, "paper_1601_08201_gb300", "csrc", "*." + e)))


def behind_short_circuit(text):
    """Lines with a collective that is (part of) the right operand of && or ||."""
    text = re.sub(r"/\*.*?\*/", lambda m: "\n" * m.group().count("\n"), text, flags=re.S)
    text = re.sub(r"//[^\n]*|\"(\\.|[^\"\\\n])*\"", "", text)
    lines = []
    for m in re.finditer(r"__\w+_sync\s*\(\s*0xffffffffu", text):
        k, depth, own = m.start() - 1, 0, True  # own: still in this operand, not past a comma at its level
        while k > 0 and text[k] not in ";{}":
            c = text[k]
            if c == ")":
                depth += 1
            elif c == "(" and depth == 0:
                own = True
            elif c == "(":
                depth -= 1
            elif depth == 0 and c == ",":
                own = False
            elif depth == 0 and own and text[k - 1:k + 1] in ("&&", "||"):
                lines.append(text.count("\n", 0, m.start()) + 1)
                break
            k -= 1
    return lines


def test_the_scan_sees_what_it_should():
    bad = "x |= a || __popc(__match_any_sync(0xffffffffu, s)) != 1;\nif (b && (c + __any_sync(0xffffffffu, d))) e();\n"
    good = "if (__any_sync(0xffffffffu, bad) && lane == 0) f(a && b, __shfl_sync(0xffffffffu, x, 0));\n" \
           "if (a || b) x = __shfl_sync(0xffffffffu, x, 0);\n"
    assert behind_short_circuit(bad) == [1, 2]
    assert behind_short_circuit(good) == []


@pytest.mark.parametrize("path", SOURCES, ids=[os.path.basename(p) for p in SOURCES])
def test_no_collective_behind_a_short_circuit(path):
    with open(path) as fh:
        assert behind_short_circuit(fh.read()) == []
