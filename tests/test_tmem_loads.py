"""tcgen05.ld is asynchronous: the registers it names hold nothing before tcgen05.wait::ld, and neither reading nor copying
them earlier is defined.  The compiler sees two unrelated statements and may copy registers between them (around a loop's
back edge, for a tied operand), so in the sources every load stands in one asm statement with its wait."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2110_09195_b200" / "csrc"
SOURCES = sorted(p.name for pattern in ("*.cu", "*.cuh", "*.h") for p in CSRC.glob(pattern))


def asm_statements(text):
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"\basm\b[^;(]*\(", text):
        quoted, depth, i = False, 1, m.end()
        while depth:
            c = text[i]
            if c == '"':
                quoted = not quoted
            elif not quoted:
                depth += (c == "(") - (c == ")")
            i += 1
        yield text[m.end():i]


@pytest.mark.parametrize("name", SOURCES)
def test_a_tensor_memory_load_is_one_statement_with_its_wait(name):
    for statement in asm_statements((CSRC / name).read_text()):
        if "tcgen05.ld" in statement:
            assert "tcgen05.wait::ld" in statement[statement.index("tcgen05.ld"):]


def test_the_loads_are_found():
    found = [s for n in SOURCES for s in asm_statements((CSRC / n).read_text()) if "tcgen05.ld" in s]
    assert found
