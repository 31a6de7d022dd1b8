"""The rule on a context's optional scratch (csrc/rec_scratch.h, host code):
the small velocity copy is kept where only the FP64 cell cache is too large."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MB, GB = 1 << 20, 1 << 30
CASES = [  # copy, cache, free -> level (0 least, 1 copy, 2 all)
    (0, 0, 0, 2),
    (1 * MB, 9 * MB, 1 * MB, 2),           # 256 MB and less without asking
    (67 * MB, 671 * MB, 200 * GB, 2),      # 256^3 FP64
    (67 * MB, 671 * MB, 3 * GB, 1),
    (67 * MB, 189 * MB, 0, 2),             # 256 MB together
    (67 * MB, 190 * MB, 0, 1),
    (67 * MB, 671 * MB, 8 * 738 * MB, 2),  # an eighth exactly
    (67 * MB, 671 * MB, 8 * 738 * MB - 8, 1),
    (537 * MB, 0, 8 * 537 * MB, 2),        # 512^3 mixed
    (537 * MB, 0, 4 * GB, 0),
    (537 * MB, 5369 * MB, 8 * GB, 1),
    (537 * MB, 5369 * MB, 1 * GB, 0),
]


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_levels(tmp_path):
    src = tmp_path / "levels.cpp"
    calls = "\n".join(f'  std::printf("%d\\n", rec::scratch_level({a}ull, {b}ull, {f}ull));' for a, b, f, _ in CASES)
    src.write_text('#include <cstdio>\n#include "rec_scratch.h"\nint main() {\n' + calls + "\n}\n")
    exe = tmp_path / "levels"
    inc = os.path.join(ROOT, "paper_2312_11448_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", inc, str(src), "-o", str(exe)], check=True)
    got = [int(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    assert got == [level for *_, level in CASES]
