"""The planes per z chunk that the library takes for the grids of the long-chunk tests of the
fused Yee update (the same header code, compiled for the host): those tests are there for
chunks longer than the ring of planes ahead, and a change of the rule must not shorten them
unnoticed."""
import os
import shutil
import subprocess

import pytest

from test_gpu_maxwell_long_chunks import CASES

HERE = os.path.dirname(os.path.abspath(__file__))


def test_long_chunks_are_long(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = tmp_path / "maxwell_planes_print"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-o", str(exe), os.path.join(HERE, "native", "maxwell_planes_print.cu")],
                   check=True)
    args, want = [], []
    for ndim, n, _, p64, p32 in CASES:
        args += [str(v) for v in (ndim, *n, 1, ndim, *n, 0)]
        want += [p64, p32]
    out = subprocess.run([str(exe), *args], capture_output=True, text=True, check=True)
    assert [int(v) for v in out.stdout.split()] == want
    assert min(want) > 4  # the ring holds 4 planes (FP32) or 3
