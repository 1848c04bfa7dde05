"""The staged kernel's variants with several sub-stages per column on the GPU against the oracle: tiles
wider than the grid, partial tiles on every axis, several tiles per CTA, two CTAs per SM; and the
default choice takes a variant that fits."""
import pytest

from paper_2004_02833_gb300 import rtpn, synth
from test_gpu_parity import assert_parity, oracle_problem

pytestmark = pytest.mark.gpu

CASES = [
    # N, shape (nz, ny, nx), bc, tile (0 = default), stage buffers
    (39, (3, 5, 88), "periodic", (80, 2, 2), 4),
    (39, (5, 3, 72), "vacuum", (72, 2, 2), 4),
    (39, (4, 3, 72), "periodic", (64, 2, 2), 5),
    (39, (3, 3, 56), "vacuum", (48, 2, 2), 7),
    (39, (7, 4, 40), "periodic", (32, 3, 3), 5),
    (29, (3, 4, 96), "vacuum", (80, 2, 2), 4),
    (29, (5, 4, 40), "periodic", (32, 3, 3), 5),
    (29, (3, 3, 72), "periodic", (64, 2, 2), 5),
    (19, (3, 5, 168), "periodic", (80, 2, 2), 4),
    (19, (5, 4, 64), "vacuum", (64, 2, 2), 5),
    (19, (3, 5, 56), "vacuum", (48, 2, 2), 4),
    (19, (4, 7, 48), "periodic", (32, 3, 3), 5),
    (15, (9, 40, 72), "periodic", (64, 2, 2), 3),  # more tiles than CTAs
    (15, (5, 6, 56), "vacuum", (48, 2, 2), 4),
    (15, (3, 5, 104), "periodic", (96, 2, 2), 4),
    (15, (6, 9, 40), "vacuum", (32, 4, 4), 3),
    (7, (9, 40, 72), "periodic", (64, 2, 2), 3),
    (7, (5, 6, 56), "vacuum", (48, 2, 2), 4),
    (7, (7, 8, 40), "periodic", (32, 3, 3), 3),
    (19, (2, 2, 8), "periodic", (0, 0, 0), 0),
    (39, (2, 1, 16), "vacuum", (0, 0, 0), 0),
]


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("N,shape,bc,tile,depth", CASES)
def test_substage_variants(cuda_device, coupling_cache, N, shape, bc, tile, depth, precision):
    inst, u0 = synth.random_instance(N, shape, seed=1200 + N, bc=bc)
    P = oracle_problem(inst, coupling_cache)
    ref = P.run(u0, 2)
    with rtpn.Context(N, inst.shape, inst.h, inst.bc, precision, inst.dt) as ctx:
        ctx.set_kernel("stage", tile, depth)
        info = ctx.info()
        assert info.kernel == 3 and (depth == 0 or (tuple(info.tile), info.depth) == (tile, depth))
        ctx.set_media(inst.sigma_a, inst.sigma_s, inst.q)
        ctx.set_moments(u0)
        ctx.step(2)
        ctx.synchronize()
        got = ctx.get_moments()
    assert_parity(got, ref, precision, P, u0, 2)
