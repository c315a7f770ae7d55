"""Host check of the factor tree's Laplace levels (csrc/minor_levels.cpp): tests/minor_levels_check.cpp
replays their words against determinants by elimination (CPU, g++)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2201_04269_gb300", "csrc")


def test_minor_levels(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    exe = str(tmp_path / "minor_levels_check")
    subprocess.run([cxx, "-O2", "-std=c++17", f"-I{CSRC}", os.path.join(ROOT, "tests", "minor_levels_check.cpp"),
                    os.path.join(CSRC, "minor_levels.cpp"), os.path.join(CSRC, "planner.cpp"), "-o", exe],
                   check=True, capture_output=True, timeout=600)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    assert out.returncode == 0 and out.stdout.startswith("OK"), out.stdout + out.stderr
