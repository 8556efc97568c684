"""Kernels that start while the kernel before them still runs (launch_overlapped) take what that
kernel, or they themselves, write with plain loads or from L2: the read-only load path is defined only
for memory that stays as it is for a kernel's whole life (source check, no GPU)."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2605_11673_gb300" / "csrc"
# the frames' and rebuilds' state: activity and claims, activity words of long units, flags of the
# zero-fill form, the frame's unit list and its count, the fixed-point sums
CHANGING = r"(?:\bustate\b|\buext\b|\bext\b|\bcflag\b|\bflags\b|\blist\b|\bcounters?\b|\bcount\b|\bS\b)"
FILES = ["sta_stream.cu", "sta_rebuild.cu", "sta_fixed.cu", "sta_fold.cuh", "sta_claim.cuh"]


def _code(name):
    return re.sub(r"//[^\n]*", "", (CSRC / name).read_text())


@pytest.mark.parametrize("name", FILES)
def test_no_read_only_loads_of_changing_words(name):
    code = _code(name)
    for m in re.finditer(r"__ldg\(", code):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(code[i], 0)
            i += 1
        arg = re.sub(r"__ld[gc]+\(.*\)", "", code[m.end():i - 1])  # not the index of another load
        assert not re.search(CHANGING, arg), f"{name}: __ldg({arg})"


@pytest.mark.parametrize("name", FILES)
def test_no_read_only_promise_on_changing_words(name):
    for m in re.finditer(r"const \w[\w ]*\*__restrict__ (\w+)", _code(name)):
        assert not re.fullmatch(CHANGING, m.group(1)), f"{name}: {m.group(0)}"
