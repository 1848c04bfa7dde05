"""The staged kernel's form for cells with h_y != h_x on the host: every y constant is the coupling times h / h_y
rounded once, and the sums are bit for bit those of a scalar loop over such constants (no shared, twice
rounded scale, whose error is the same for every y term)."""
import os
import subprocess

import pytest

from test_fused_host import CSRC, HERE, ROOT, _nvcc

VARIANTS = [(7, 32, 3, 3, 3, 1), (15, 64, 2, 2, 3, 2), (19, 80, 2, 2, 4, 2), (39, 80, 2, 2, 4, 4)]


@pytest.mark.parametrize("variant", VARIANTS)
def test_scaled_sweep_is_a_scalar_loop_bit_for_bit(tmp_path, variant):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "check_scaled")
    names = ("SN", "STX", "STY", "STZ", "SNB", "SEM")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "-diag-suppress", "20011,20013,20015",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC] + [f"-DRTPN_{n}={v}" for n, v in zip(names, variant)] + [
           os.path.join(HERE, "host", "check_scaled.cu"), os.path.join(CSRC, "model.cpp"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]
    for sy, sz in ((1.0, 1.0), (1 / 1.3, 1 / 1.7), (1 / 1.7, 1.0), (0.6, 0.9), (1.25, 1.0), (1 / 1.1, 1 / 1.1)):
        r = subprocess.run([exe, repr(sy), repr(sz), "5"], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-500:]
        seen, bad, plain = map(int, r.stdout.split())
        assert seen > 100 and bad == 0, (sy, sz, seen, bad)
        assert (plain == 0) == (sy == 1.0)
