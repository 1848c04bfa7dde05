"""The generic kernel's compiled FP64 form (orders 1 to 9, cubic cells) against the oracle: single cells, rows
shorter and longer than a warp, grids of one-warp and of full blocks, both boundaries, half and full
passes; orders and cells without it (table kernel) beside it."""
import numpy as np
import pytest

from paper_2004_02833_gb300 import rtpn, synth
from test_gpu_parity import oracle_problem

pytestmark = pytest.mark.gpu

CASES = [(N, shape, bc) for N in (1, 3, 5, 7, 9) for shape, bc in
         (((1, 1, 1), "periodic"), ((2, 3, 5), "vacuum"), ((3, 5, 33), "periodic"), ((4, 2, 65), "vacuum"))]
CASES += [(3, (54, 54, 54), "periodic"), (2, (3, 4, 5), "periodic"), (4, (3, 4, 5), "vacuum")]


@pytest.mark.parametrize("N,shape,bc", CASES)
def test_fp64_passes_vs_oracle(cuda_device, coupling_cache, N, shape, bc):
    inst, u0 = synth.random_instance(N, shape, seed=1500 + N, bc=bc)
    P = oracle_problem(inst, coupling_cache)
    with rtpn.Context(N, shape, inst.h, bc, "fp64", inst.dt) as ctx:
        assert ctx.info().kernel == 1
        ctx.set_media(inst.sigma_a, inst.sigma_s, inst.q)
        ctx.set_moments(u0)
        ctx.substep(1, half=True)
        ref = P.substep(u0, 1, 0.5 * inst.dt)
        assert np.abs(ctx.get_moments() - ref).max() <= 1e-12 * np.abs(ref).max()
        ctx.substep(0)
        ref = P.substep(ref, 0, inst.dt)
        assert np.abs(ctx.get_moments() - ref).max() <= 1e-12 * np.abs(ref).max()
        ctx.step(2)
        ref = P.run(ref, 2)
        assert np.abs(ctx.get_moments() - ref).max() <= 1e-12 * np.abs(ref).max()
