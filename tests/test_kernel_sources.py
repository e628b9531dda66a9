"""Properties of the kernel sources that no run on a GPU can be relied on to show."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2206_00470_gb300", "csrc")
READ_ONLY = re.compile(r"__ldg\s*\(|\bld\.global\.nc\b|const\s[\w\s]*\*\s*__restrict__")


def _code(text):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def _kernels(code):
    """(name, signature and body) of every kernel of a source, and the text outside them."""
    out, rest, at = [], [], 0
    for m in re.finditer(r"__global__", code):
        begin = code.index("{", m.start())
        depth, i = 1, begin + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            i += 1
        text = code[m.start():i]
        out.append((re.search(r"(\w+)\s*\((?:Store|SortArgs|SmallArgs|Sel|const|int32_t|uint32_t)\b", text).group(1), text))
        rest.append(code[at:m.start()])
        at = i
    return out, "".join(rest) + code[at:]


def test_overlapping_kernels_read_with_plain_loads():
    """A kernel launched while the one before it drains (it begins with after_previous()) runs from before that
    one's last writes: loads that promise unchanging data may be moved in front of its wait."""
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        kernels, rest = _kernels(_code(open(path).read()))
        for name, text in kernels:
            if "after_previous()" in text:
                seen += 1
                assert not READ_ONLY.search(text), f"{os.path.basename(path)}: {name}"
        # (device functions, which such kernels may call)
        assert not READ_ONLY.search(rest), os.path.basename(path)
    assert seen >= 12
