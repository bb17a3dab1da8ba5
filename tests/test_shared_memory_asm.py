"""Inline assembly that reads or writes shared memory is tied to its place: an
asm statement without volatile and a "memory" clobber is, to the compiler, a
function of its operands, which it may move across __syncthreads, so that a read
could come before the stores of other threads that the barrier orders."""
import pathlib
import re

import pytest

import paper_2609_37693_gb300 as oz

CSRC = pathlib.Path(oz.__file__).parent / "csrc"
SOURCES = sorted(p for p in CSRC.iterdir() if p.suffix in (".cu", ".cuh", ".cpp", ".h"))


def _statements(text):
    """(asm statement up to its closing parenthesis, line) of a source."""
    for m in re.finditer(r"\basm\b\s*(volatile\s*)?\(", text):
        depth, i, quoted = 1, m.end(), False
        while depth:
            c = text[i]
            if quoted:
                i += c == "\\"
                quoted = c != '"'
            elif c == '"':
                quoted = True
            else:
                depth += (c == "(") - (c == ")")
            i += 1
        yield text[m.start():i], text.count("\n", 0, m.start()) + 1


@pytest.mark.parametrize("path", SOURCES, ids=lambda p: p.name)
def test_asm_on_shared_memory_stays_in_place(path):
    text = re.sub(r"//[^\n]*", "", path.read_text())
    for asm, line in _statements(text):
        if re.search(r"\b(ld|st|atom|red)(\.[a-z]+)*\.shared", asm):
            assert "volatile" in asm and asm.rstrip(" )").endswith('"memory"'), f"{path.name}:{line}: {asm}"
