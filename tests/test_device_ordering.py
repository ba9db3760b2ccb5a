"""Orders that the device code states to the compiler, checked in its source: nothing
else in the language keeps memory accesses on their side of an inline assembly statement."""
import pathlib
import re

import pytest

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


# Pointers that a kernel only writes may be __restrict__; one that it reads after a wait may not.
WRITTEN_ONLY = {"Mout", "dst", "sdst", "partial", "lpart", "grad", "out", "loss", "wmat"}


@pytest.mark.parametrize("name", sorted(f.name for f in CSRC.glob("*.cu")))
def test_overlapped_kernels_read_nothing_through_restrict(name):
    """A kernel that waits for its stream predecessor starts while that one still writes:
    what it reads is not promised to be unwritten."""
    text = _code(name)
    found = 0
    for m in re.finditer(r"\bvoid\s+(?:__launch_bounds__\s*\([^{;]*?\)\s*)?(\w+)\s*\(", text):
        params = _balanced(text, m.end() - 1)
        rest = text[m.end() - 1 + len(params):].lstrip()
        if not rest.startswith("{"):
            continue
        body = _balanced(rest, 0, "{}")
        if "wait_for_predecessor();" not in body:
            continue
        found += 1
        for const, var in re.findall(r"(const\s+)?[\w:]+\s*\*\s*__restrict__\s+(\w+)", params + body):
            assert not const, (m.group(1), var)
            assert var in WRITTEN_ONLY, (m.group(1), var)
    if name in ("tfkt_fused.cu", "tfkt_lpm.cu", "tfkt_mlp.cu", "tfkt_split.cu"):
        assert found >= 2


@pytest.mark.parametrize("name", sorted(f.name for f in CSRC.glob("*.cu")))
def test_copies_are_ordered_on_a_stream(name):
    """A blocking cudaMemcpy or cudaMemset is ordered against the default stream only, and from
    pageable memory it may return before the data has arrived: a kernel on a non-blocking
    stream may then run without it."""
    assert not re.findall(r"\bcuda(?:Memcpy|Memset|Memcpy2D)\s*\(", _code(name))
