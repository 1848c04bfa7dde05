"""The TMA-staged kernel with several sub-stages per column, compiled for the host (nvcc, no GPU) and run
over bounds-checked memory, one pass against the oracle's substep: columns that start inside a
sub-stage and at its edge, both classes (class 1 finishes one slot behind its sources), partial tiles,
wrapped and zero-filled halos, scaled y differences, FP32 and BF16 storage."""
import os
import subprocess

import numpy as np
import pytest

from oracle import stepper as st
from paper_2004_02833_gb300 import synth

from test_fused_host import CSRC, HERE, ROOT, _bf16_round, _nvcc

VARIANTS = {  # (order, tile x, y, z, stage buffers, sub-stages), entries of stage_variants.h
    "39": (39, 80, 2, 2, 4, 4),
    "39w": (39, 32, 3, 3, 5, 4),
    "19": (19, 64, 2, 2, 5, 2),
    "15": (15, 64, 2, 2, 3, 2),
}
CASES = [
    # variant, shape (nz, ny, nx) with nx a multiple of 8, bc, target class, half step, storage, CTAs, h/h_y
    ("39", (3, 3, 88), "periodic", 0, 0, "fp32", 2, 1.0),
    ("39", (2, 3, 72), "vacuum", 1, 1, "bf16", 1, 1.0),
    ("39w", (4, 3, 40), "periodic", 1, 0, "fp32", 2, 1.0),
    ("19", (3, 5, 72), "periodic", 1, 0, "fp32", 3, 0.8),
    ("19", (4, 4, 64), "vacuum", 0, 0, "bf16", 2, 1.0),
    ("15", (5, 3, 136), "vacuum", 0, 0, "fp32", 2, 0.6),
    ("15", (4, 5, 64), "periodic", 1, 1, "fp32", 5, 1.0),
    ("15", (1, 1, 8), "periodic", 1, 0, "fp32", 1, 1.0),
]


@pytest.fixture(scope="module")
def emulators(tmp_path_factory):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("substage_host")
    out = {}
    for key, (n, tx, ty, tz, nb, ch) in VARIANTS.items():
        exe = str(d / f"emulate_substage_{key}")
        cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O1", "-diag-suppress", "20011",
               "-I", os.path.join(ROOT, "include"), "-I", CSRC, f"-DRTPN_SN={n}", f"-DRTPN_STX={tx}",
               f"-DRTPN_STY={ty}", f"-DRTPN_STZ={tz}", f"-DRTPN_SNB={nb}", f"-DRTPN_SEM={ch}",
               os.path.join(HERE, "host", "emulate_substage.cu"), os.path.join(CSRC, "model.cpp"), "-o", exe]
        res = subprocess.run(cmd, capture_output=True, text=True)
        assert res.returncode == 0, res.stderr[-2000:]
        out[key] = exe
    return out


@pytest.mark.parametrize("key,shape,bc,cls,half,prec,ctas,sy", CASES)
def test_substages_on_host_vs_oracle(emulators, tmp_path, key, shape, bc, cls, half, prec, ctas, sy):
    N = VARIANTS[key][0]
    inst, u = synth.random_instance(N, shape, seed=1100 + N, bc=bc)
    nz, ny, nx = shape
    fin, fout = str(tmp_path / "in.bin"), str(tmp_path / "out.bin")
    np.concatenate([u.ravel(), inst.sigma_a.ravel(), inst.sigma_s.ravel(), inst.q.ravel()]).tofile(fin)
    res = subprocess.run([emulators[key], str(cls), str(nx), str(ny), str(nz), str(0 if bc == "periodic" else 1),
                          repr(inst.h), repr(inst.dt), str(half), prec, str(ctas), fin, fout, repr(sy)],
                         capture_output=True, text=True, timeout=600)
    assert res.returncode == 0, res.stderr[-2000:]
    got = np.fromfile(fout).reshape(u.shape)
    P = st.Problem(N, inst.sigma_a, inst.sigma_s, inst.q, (inst.h, inst.h / sy, inst.h), inst.dt, bc)
    u_in = u.astype(np.float32).astype(np.float64) if prec == "fp32" else _bf16_round(u)
    ref = P.substep(u_in, cls, 0.5 * inst.dt if half else inst.dt)
    assert np.isfinite(got).all()
    if prec == "fp32":
        assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()
    else:  # one pass rounds its class once: within one BF16 ulp (2^-8 relative) of the oracle
        m = P.cls == cls
        assert np.all(np.abs(got[m] - ref[m]) <= 2.0 ** -8 * np.abs(ref[m]) + 1e-6 * np.abs(ref).max())
        assert np.array_equal(got[~m], u_in[~m])
