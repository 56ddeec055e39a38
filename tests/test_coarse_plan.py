"""The plan of the coarse launch (csrc/coarse_plan.h, built here for the host):
divisions by multiplication are exact over every index they are used for, the
grids of all levels lie apart in shared memory, slabs tile the grids, and the
face slots are distinct and inside, over box sizes, blocks of root boxes,
forests and both precisions."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_plans(tmp_path):
    exe = str(tmp_path / "coarse_plan_host")
    subprocess.run(["g++", "-O1", "-std=c++17", "-o", exe, os.path.join(ROOT, "tests", "coarse_plan_host.cpp")],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert int(out[0]) > 500 and out[1] == "0", out
