"""The compiled FP64 kernel's threads: every cell once, and no more warps than cells call for, whatever the row
length (rows of 1 to 140 cells; with one warp per row of 33 cells half the FP64 work would be for idle lanes)."""
import os
import subprocess

import pytest

from test_fused_host import CSRC, HERE, ROOT, _nvcc


def test_lanes_are_filled_whatever_the_row_length(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "check_lanes64")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "-diag-suppress", "20011,20013,20015",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC, os.path.join(HERE, "host", "check_lanes64.cu"),
           os.path.join(CSRC, "model.cpp"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-500:])
    # rows folded into the warp leave the last warp's lanes idle: 96 for 65 cells at worst; tiles at most a tenth
    assert float(r.stdout) <= 1.5
