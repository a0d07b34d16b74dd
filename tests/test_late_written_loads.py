"""Loads through the read-only path (ld.global.nc, __ldg) are defined only for memory that nothing writes while the kernel lives.  A
programmatic dependent lives while the kernel before it still writes: the activations, and in the no-allocation call the scales.  So what such
a launch of the tensor-core kernel reads that way is only what was written when its group was created; chains are no dependents."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2110_09195_b200" / "csrc"
# descriptions and ranks of a group, thresholds of its signs, dependencies of a chain
CREATED = {"p",   # g_ld, for chains
           "src + i", "p.ranks + (size_t)rank * G + blockIdx.x", "L.threshold + c", "deps + fdiv((uint32_t)tile, dCt)"}


def _arguments(text, call):
    for m in re.finditer(r"\b%s\(" % re.escape(call), text):
        depth, i = 1, m.end()
        while depth:
            depth += (text[i] == "(") - (text[i] == ")")
            i += 1
        yield text[m.end():i - 1]


def test_the_read_only_path_is_for_what_was_written_at_creation():
    text = re.sub(r"//[^\n]*", "", (CSRC / "snn_tcg.cu").read_text() + (CSRC / "snn_tc_common.cuh").read_text())
    assert set(_arguments(text, "__ldg")) == CREATED
    assert "const uint32_t* src = reinterpret_cast<const uint32_t*>(p.layers);" in text   # (what "src + i" is)
    assert "return LATE ? *p : __ldg(p);" in text and "constexpr bool LATE = !CHAIN && !TAGGED;" in text
    assert set(_arguments(text, "g_ld<LATE>")) == {"q", "L.alpha + c"} and not re.search(r"\bg_ld<(?!LATE)", text)
    assert ".nc" not in "".join(re.findall(r'"[^"\n]*"', text))


def test_no_parameter_of_the_launches_dependents_promises_read_only_memory():
    """const __restrict__ pointers may be read through that path by the compiler's choice."""
    text = (CSRC / "snn_tcg.cu").read_text()
    for kernel in ("tcg_conv_kernel", "g_static_weights_kernel"):
        head = text[text.index(f" {kernel}("):]
        head = head[:head.index("{")]
        assert not re.search(r"const\s+\w+\s*\*\s*__restrict__", head)
