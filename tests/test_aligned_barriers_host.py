"""Barrier instructions written out in the kernels are the aligned forms, which a whole warp has to
execute together: each stands right behind a __syncwarp() (source check, no GPU)."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2605_11673_gb300" / "csrc"


def test_warps_are_whole_at_aligned_barriers():
    found = 0
    for f in sorted(CSRC.glob("*.cu*")):
        code = re.sub(r"//[^\n]*", "", f.read_text())
        for m in re.finditer(r'asm volatile\(\s*"(?:barrier\.|bar\.)', code):
            found += 1
            assert re.search(r"__syncwarp\(\);\s*$", code[:m.start()]), f"{f.name}: {code[m.start():m.end() + 40]}"
    assert found >= 3
