"""The shared memory of the coarse launch (csrc/coarse_plan.h, built here for the
host), with and without variable coefficients: the coefficient arrays lie apart
from the grids and from each other and are copied in whole 16-byte pieces, the
correction's scratch holds the largest level that uses it, and every block's slab
touches no more boxes than it has entries for."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_layouts(tmp_path):
    exe = str(tmp_path / "coarse_plan_layout_host")
    subprocess.run(["g++", "-O1", "-std=c++17", "-o", exe, os.path.join(ROOT, "tests", "coarse_plan_layout_host.cpp")],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert int(out[0]) > 1000 and out[1] == "0", out
