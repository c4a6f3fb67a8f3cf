"""The digit planes' storage and box coordinates as the library computes them (csrc/digit_planes.h),
compiled for the host and compared with what the MMA operand reads (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2505_03755_gb300", "csrc")


def _run(tmp_path, include):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "digit_planes")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror", "-Wno-unused-function",
                    "-I", include, os.path.join(ROOT, "tests", "digit_planes.cc"), "-o", exe],
                   check=True)
    return subprocess.run([exe], capture_output=True, text=True)


def test_boxes_hold_what_the_products_need(tmp_path):
    r = _run(tmp_path, CSRC)
    assert r.returncode == 0, r.stdout
    assert r.stdout.startswith("ok ") and int(r.stdout.split()[1]) > 1_000_000


@pytest.mark.parametrize("old,new", [
    ("(int)(r & 4) << 1", "(int)(r & 2) << 2"),                       # another row's halves swapped
    ("(row0 % ROWGRAN)", "(row0 % 8)"),                               # start between two box rows
    ("(b.r + ROWGRAN - 1) / ROWGRAN * ROWGRAN : b.r", "b.r : b.r"),   # ragged rows not padded
    ("8L * nb1 * BK", "8L * BK"),                                     # ragged K blocks
    ("J * (J + 1) / 2) * 8", "J * (J - 1) / 2) * 8"),                 # another stored tile
])
def test_a_wrong_layout_is_found(tmp_path, old, new):
    src = open(os.path.join(CSRC, "digit_planes.h")).read()
    assert src.count(old) == 1
    (tmp_path / "digit_planes.h").write_text(src.replace(old, new))
    assert _run(tmp_path, str(tmp_path)).returncode != 0
