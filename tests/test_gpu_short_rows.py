"""Short rows padded to whole sectors (FP32 below 40 cells): steps against the oracle at every remainder."""
import pytest

from paper_2004_02833_gb300 import rtpn, synth
from test_gpu_parity import assert_parity, oracle_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [9, 11, 14, 17, 18, 19, 25, 27, 31, 33, 35, 37, 41])
@pytest.mark.parametrize("bc", ["periodic", "vacuum"])
def test_steps_on_short_padded_rows(cuda_device, coupling_cache, nx, bc):
    inst, u0 = synth.random_instance(15, (3, 5, nx), seed=1600 + nx, bc=bc)
    P = oracle_problem(inst, coupling_cache)
    ref = P.run(u0, 2)
    with rtpn.Context(15, inst.shape, inst.h, bc, "fp32", inst.dt) as ctx:
        assert ctx.info().kernel == 3 and ctx.info().state_bytes > 256 * 3 * 5 * nx * 4
        ctx.set_media(inst.sigma_a, inst.sigma_s, inst.q)
        ctx.set_moments(u0)
        ctx.step(2)
        ctx.set_kernel("window")  # and back to dense rows
        got = ctx.get_moments()
    assert_parity(got, ref, "fp32", P, u0, 2)
