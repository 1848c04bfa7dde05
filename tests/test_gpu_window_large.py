"""Window and batched passes on grids whose data do not stay in L2, where a tile asks for its rows first (orders 5,
7 and 9): odd extents, both boundaries, non-cubic cells, per-order factors and both storages against the
generic kernel, which the oracle tests cover."""
import pytest
import torch

from paper_2004_02833_gb300 import rtpn

pytestmark = pytest.mark.gpu

FP32 = 2e-5  # two FP32 results, each within 1e-5 of the oracle (times max |u|)
CASES = [
    # N, shape (nz, ny, nx), bc, storage, option; 104 to 125 MB of state and factors each
    (5, (79, 77, 79), "periodic", "fp32", None),
    (5, (89, 91, 93), "vacuum", "bf16", "spacing"),
    (7, (67, 70, 73), "vacuum", "fp32", None),
    (7, (63, 65, 65), "periodic", "bf16", "aniso"),
    (9, (61, 59, 63), "periodic", "fp32", "spacing"),
    (9, (53, 55, 57), "vacuum", "fp32", "aniso"),
    (9, (75, 73, 77), "vacuum", "bf16", None),
]


def fill(nc, shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.randn((nc,) + shape, generator=g, device="cuda")
    return u, torch.rand((3,) + shape, generator=g, device="cuda", dtype=torch.float64)


def check(got, ref, precision):
    top = ref.abs().max()
    if precision == "fp32":
        assert (got - ref).abs().max() <= FP32 * top
    else:  # a pass rounds its class once: a rounding may tip the other way by one BF16 ulp
        assert ((got - ref).abs() <= 2.0 ** -7 * ref.abs() + FP32 * top).all()


@pytest.mark.parametrize("N,shape,bc,precision,option", CASES)
def test_window_passes_on_large_grids(cuda_device, N, shape, bc, precision, option):
    u, m = fill((N + 1) ** 2, shape, 70 + N)
    got, ref = torch.empty_like(u), torch.empty_like(u)
    ctxs = []
    for kernel in ("window", "generic"):
        ctx = rtpn.Context(N, shape, 0.1, bc, precision)
        ctx.set_kernel(kernel)
        if option == "spacing":
            ctx.set_spacing(0.1, 0.13, 0.17)
        if option == "aniso":
            ctx.set_scattering([0.8 ** l for l in range(N + 1)])
        ctx.set_media(m[0], m[1], m[2])
        ctxs.append(ctx)
    a, b = ctxs
    a.set_moments(u)
    with a, b:
        for cls, half in ((1, True), (0, False)):
            a.get_moments(got)
            a.synchronize()
            b.set_moments(got)  # both from the same state
            a.substep(cls, half)
            b.substep(cls, half)
            a.get_moments(got)
            b.get_moments(ref)
            a.synchronize()
            b.synchronize()
            check(got, ref, precision)


def test_batch_whose_instances_together_leave_l2(cuda_device):
    # grouped passes against the same instances stepped one by one in the batch (looped form), each of which
    # alone would stay in L2
    inst = [(N, (n, n + 1, n + 2), 0.1, bc, None) for N, n, bc in
            ((9, 41, "periodic"), (9, 37, "vacuum"), (7, 49, "vacuum"), (7, 45, "periodic"), (5, 55, "periodic"), (5, 51, "vacuum"), (9, 40, "vacuum"))]
    outs = []
    for looped in (False, True):
        batch = rtpn.Batch(inst)
        res = []
        for i, (N, shape, *_) in enumerate(inst):
            u, m = fill((N + 1) ** 2, shape, 80 + i)
            batch[i].set_media(m[0], m[1], m[2])
            batch[i].set_moments(u)
            batch[i].synchronize()
            res.append(u)
        (batch.step_looped if looped else batch.step)(2)
        batch.synchronize()
        for i, u in enumerate(res):
            batch[i].get_moments(u)
            batch[i].synchronize()
        outs.append(res)
    for x, y in zip(*outs):
        assert (x - y).abs().max() <= 1e-6 * y.abs().max()  # the same body, compiled twice
