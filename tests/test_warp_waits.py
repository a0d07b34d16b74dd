"""A shuffle orders no memory: where one lane waits for a phase and shuffles its answer, what it has seen is not the other lanes'.  The table
warp and the expanders write, with all lanes, over what the phase says has been read, so every lane looks for itself."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2110_09195_b200" / "csrc"


def _body(text, start):
    i = text.index("{", text.index(start))
    depth, j = 1, i + 1
    while depth:
        depth += (text[j] == "{") - (text[j] == "}")
        j += 1
    return text[i + 1:j - 1]


def test_every_lane_of_a_whole_warp_wait_looks_for_itself():
    text = re.sub(r"//[^\n]*", "", (CSRC / "snn_tcg.cu").read_text())
    body = _body(text, "auto wait_phase =")
    assert "__all_sync(0xffffffffu, mbar_test(bar, parity))" in body
    assert "const bool over = __all_sync(0xffffffffu, !*abort_flag && mbar_wait_backoff(bar, parity, ns));" in body
    assert "__shfl" not in body and "lane == 0" not in body[:body.index("const bool over")]
