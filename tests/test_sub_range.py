"""The particle kernel finds a slot's source sub-range by a walk through the tile's source
table.  The walk (the same header code, compiled for the host) is checked against a linear
search, and on tables that do not hold the slot, as a recorded device error can leave them:
there it must stay inside the table."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_walk_finds_the_sub_range_and_stays_in_the_table(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "sub_range_check"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-o", str(exe), os.path.join(HERE, "native", "sub_range_check.cu")],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
