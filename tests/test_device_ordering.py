"""Orders that the device code states to the compiler, checked in its source: nothing
else in the language keeps memory accesses on their side of an inline assembly statement."""
import pathlib
import re

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2201_10132_gb300" / "csrc"


def _code(name):
    return re.sub(r"//[^\n]*", "", (CSRC / name).read_text())


def _balanced(text, start, pair="()"):
    """The text from the opening bracket at `start` to its closing one."""
    depth, quoted = 0, False
    for k in range(start, len(text)):
        c = text[k]
        if c == '"':
            quoted = not quoted
        elif not quoted:
            depth += (c == pair[0]) - (c == pair[1])
            if depth == 0:
                return text[start:k + 1]
    raise AssertionError("unbalanced")


def test_tensor_core_statements_clobber_memory():
    """tcgen05, mbarrier, fence and barrier statements: operand stores stay in front of them."""
    text = _code("tfkt_umma.cuh")
    asm = [_balanced(text, m.end() - 1) for m in re.finditer(r"\basm volatile\(", text)]
    assert len(asm) >= 12
    assert not [a for a in asm if '"memory"' not in a]


def test_tensor_memory_load_and_its_wait_are_one_statement():
    text = _code("tfkt_umma.cuh")
    loads = [a for a in (_balanced(text, m.end() - 1) for m in re.finditer(r"\basm volatile\(", text))
             if "tcgen05.ld." in a]
    assert loads and all("tcgen05.wait::ld" in a for a in loads)
