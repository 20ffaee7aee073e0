"""Field read-outs queue their copies into the caller's memory and wait once at the end.  When
one of them cannot be queued the call must still wait for those before it: checked on the
host, with a fake queue that fails at each item."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_a_failed_item_still_waits_for_those_before_it(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "queue_wait_check"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-o", str(exe), os.path.join(HERE, "native", "queue_wait_check.cu")],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
