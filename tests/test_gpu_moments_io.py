"""Full states in and out on the device (one kernel over all components) against the per-component calls:
rows of whole 16-byte groups and odd ones, unaligned caller buffers, every storage and caller type."""
import pytest
import torch

from paper_2004_02833_gb300 import rtpn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 8, 16), (3, 5, 7), (1, 1, 1), (2, 3, 682), (9, 17, 31)])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("offset", [0, 1])
def test_moments_on_device_equal_components(cuda_device, shape, precision, dtype, offset):
    N, nc, V = 3, 16, shape[0] * shape[1] * shape[2]
    g = torch.Generator(device="cuda").manual_seed(5)
    store = torch.empty(nc * V + 1, dtype=dtype, device="cuda")
    u = store[offset:offset + nc * V].view((nc,) + shape)
    u.copy_(torch.randn((nc,) + shape, generator=g, dtype=dtype, device="cuda"))
    with rtpn.Context(N, shape, 0.1, "periodic", precision) as a, rtpn.Context(N, shape, 0.1, "periodic", precision) as b:
        a.set_moments(u)
        for c in range(nc):
            b.set_component(c, u[c].clone())
        back = torch.empty(nc * V + 1, dtype=dtype, device="cuda")[offset:offset + nc * V].view((nc,) + shape)
        assert a.get_moments(back) is back
        one = torch.empty(shape, dtype=dtype, device="cuda")
        for c in range(nc):
            a.get_component(c, one)
            torch.cuda.synchronize()
            assert torch.equal(one, back[c])  # set_moments, read by component, and get_moments
            b.get_component(c, one)
            torch.cuda.synchronize()
            assert torch.equal(one, back[c])  # the same values as set by component
