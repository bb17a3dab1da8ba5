"""Kernels that may be launched while the kernel before them on the stream still
runs (launch_kernel of oz_launch.h) wait for it: each of them calls pdl_wait, and
lets its own successor start only after that. A kernel without the wait, launched
so, would race with its predecessor; every launch of the sources is checked."""
import pathlib
import re

import paper_2609_37693_gb300 as oz

CSRC = pathlib.Path(oz.__file__).parent / "csrc"
TEXT = {p.name: re.sub(r"//[^\n]*", "", p.read_text()) for p in sorted(CSRC.glob("*.cu*"))}


def _block(text, start, opening, closing):
    i = text.index(opening, start)
    depth = 0
    for j in range(i, len(text)):
        depth += (text[j] == opening) - (text[j] == closing)
        if depth == 0:
            return text[i:j + 1], j + 1
    raise AssertionError("unbalanced source")


def _kernels():
    out = {}
    for text in TEXT.values():
        for m in re.finditer(r"__global__", text):
            name = re.search(r"\b(\w+_kernel)\s*\(", text[m.end():])
            _, after = _block(text, m.end() + name.end() - 1, "(", ")")
            out[name.group(1)] = _block(text, after, "{", "}")[0]
    return out


def _launched_dependent():
    """(source, kernel names) of each launch through launch_kernel."""
    for src, text in TEXT.items():
        for m in re.finditer(r"\blaunch_kernel\(", text):
            call = _block(text, m.start(), "(", ")")[0]
            names = re.findall(r"\b(\w+_kernel)\b", call)
            if not names:                                  # a variable: what it was set from
                at = text.rindex("auto kernel =", 0, m.start())
                names = re.findall(r"\b(\w+_kernel)\b", text[at:text.index(";", at)])
            yield src, names


def test_dependent_kernels_wait_for_their_predecessor():
    kernels, launches = _kernels(), list(_launched_dependent())
    assert len(launches) >= 5 and all(names for _, names in launches)
    for src, names in launches:
        for name in names:
            body = kernels[name]
            assert body.count("pdl_wait();") == 1 and body.count("pdl_trigger();") == 1, (src, name)
            assert body.index("pdl_wait();") < body.index("pdl_trigger();"), (src, name)


def test_the_launch_attribute_is_set_in_one_place():
    uses = [p.name for p in CSRC.iterdir() if p.suffix in (".cu", ".cuh", ".h", ".cpp")
            and "ProgrammaticStreamSerialization" in re.sub(r"//[^\n]*", "", p.read_text())]
    assert uses == ["oz_launch.h"]


def test_no_launch_helper_is_left_without_a_caller():
    """Helpers of oz_launch.h that nothing calls would be a second way to launch."""
    head = re.sub(r"//[^\n]*", "", (CSRC / "oz_launch.h").read_text())
    for name in re.findall(r"inline [\w ]+?\b(\w+)\(", head):
        calls = sum(len(re.findall(rf"\b{name}\(", t)) for t in TEXT.values())
        assert calls > 0, name
