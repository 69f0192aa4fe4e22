"""The tile count of a row block (csrc/layout.cuh) on the host, up to the
planner's largest block height of 2^31 - 1 rows: a count formed in fewer bits
than it needs leaves tiles out, and the block's R is then not A's.  No GPU."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1301_1071_gb300", "csrc")


def test_row_tiles(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "row_tiles")
    subprocess.run([gxx, "-std=c++17", "-O1", "-ftrapv", "-Wall", "-I", CSRC, "-o", exe,
                    os.path.join(ROOT, "tests", "host", "row_tiles.cpp")], check=True)
    top = 2**31 - 1
    cases = [(r, B, bt) for B, bt in [(128, 128), (320, 312), (640, 614), (1024, 1), (2048, 2047)]
             for r in [1, 2, B - 1, B, B + 1, B + bt, B + bt + 1, 100_003, top - B, top - 128, top - 127, top - 1, top]]
    out = subprocess.run([exe], input="".join(f"{r} {B} {bt}\n" for r, B, bt in cases), capture_output=True,
                         text=True, check=True, timeout=60).stdout.split()
    assert [int(x) for x in out] == [1 + max(0, -(-(r - B) // bt)) for r, B, bt in cases]


def test_panel_kernel_takes_its_tiles_from_it():
    """The panel form's block height limit is the planner's (2^31 - 1 rows), so its
    count is row_tiles', with no sum of rows and a tile in int."""
    src = open(os.path.join(CSRC, "panel64.cuh")).read()
    assert re.search(r"ntiles = row_tiles\(rows, TR, TR\)", src)
    assert not re.search(r"\(rows \+ TR", src)
