"""The staged kernel's tiles by ticket on grids where every CTA takes at least six of them (past the four-entry
ring that hands the tiles on): one variant of each order in both storages, passes in a row (the counters
start from zero again), the adjoint, contexts side by side on two streams, and cells with h_y != h_x.
The reference is the generic kernel, which the oracle tests cover."""
import numpy as np
import pytest
import torch

from paper_2004_02833_gb300 import rtpn, synth

pytestmark = pytest.mark.gpu

VARIANTS = [(7, (64, 2, 2), 3), (15, (64, 2, 2), 3), (19, (80, 2, 2), 4), (29, (80, 2, 2), 4), (39, (80, 2, 2), 4)]
FP32 = 2e-5  # two FP32 results, each within 1e-5 of the oracle (times max |u|)


def many_tiles(tile):
    """nz, ny of a grid of one tile column with at least six tiles per CTA (at most two CTAs per SM)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    side = 2
    while (side // tile[1]) * (side // tile[2]) < 6 * 2 * sms:
        side += 2
    return side + 1, side  # a partial tile in z


def pair(N, shape, precision, tile, depth, bc="periodic", spacing=None, seed=60):
    """The same problem on the staged and on the generic kernel, and its state (float32, on the device)."""
    inst, _ = synth.random_instance(min(N, 7), shape, seed=seed, bc=bc)
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.randn(((N + 1) ** 2,) + shape, generator=g, dtype=torch.float32, device="cuda")
    out = []
    for kernel in ("stage", "generic"):
        ctx = rtpn.Context(N, shape, inst.h, bc, precision, inst.dt)
        ctx.set_kernel(kernel, tile if kernel == "stage" else (0, 0, 0), depth if kernel == "stage" else 0)
        if spacing:
            ctx.set_spacing(*(s * inst.h for s in spacing))
        ctx.set_media(inst.sigma_a, inst.sigma_s, inst.q)
        ctx.set_moments(u)
        out.append(ctx)
    assert tuple(out[0].info().tile) == tile and out[0].info().kernel == 3
    return out[0], out[1], u


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("N,tile,depth", VARIANTS)
@pytest.mark.parametrize("spacing", [None, (1.0, 1.3, 1.7)])
def test_passes_in_a_row(cuda_device, N, tile, depth, precision, spacing):
    nz, ny = many_tiles(tile)
    shape = (nz, ny, 8)
    a, b, u = pair(N, shape, precision, tile, depth, spacing=spacing)
    got, ref = torch.empty_like(u), torch.empty_like(u)
    with a, b:
        for cls, half in ((1, True), (0, False), (1, False), (0, False)):
            a.get_moments(got)
            a.synchronize()
            b.set_moments(got)  # both from the same state
            a.substep(cls, half)
            b.substep(cls, half)
            a.get_moments(got)
            b.get_moments(ref)
            a.synchronize()
            b.synchronize()
            top = ref.abs().max()
            if precision == "fp32":
                assert (got - ref).abs().max() <= FP32 * top
            else:  # the pass rounds its class once: a rounding may tip the other way by one BF16 ulp
                assert ((got - ref).abs() <= 2.0 ** -7 * ref.abs() + FP32 * top).all()


def test_adjoint_on_many_tiles(cuda_device):
    N, tile, depth = VARIANTS[1]
    nz, ny = many_tiles(tile)
    a, b, u = pair(N, (nz, ny, 8), "fp32", tile, depth, bc="vacuum")
    w = np.random.default_rng(61).uniform(0.0, 1.0, (nz, ny, 8))
    with a, b:
        Ja, ga = a.adjoint(w, 2, ckpt_every=1)
        Jb, gb = b.adjoint(w, 2, ckpt_every=1)
    # both within 1e-4 of the oracle's discrete adjoint (the FP32 bound of the adjoint tests)
    assert abs(Ja - Jb) <= 2e-4 * abs(Jb)
    for x, y in zip(ga, gb):
        assert np.abs(x - y).max() <= 2e-4 * np.abs(y).max()


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_contexts_side_by_side_on_two_streams(cuda_device, precision):
    # each context has its own counters: the results are those of the same steps alone, bit for bit
    N, tile, depth = VARIANTS[1]
    nz, ny = many_tiles(tile)
    ctxs = [pair(N, (nz, ny, 8 + 8 * i), precision, tile, depth, seed=62 + i) for i in range(2)]
    streams = [torch.cuda.Stream() for _ in ctxs]
    alone = []
    for (a, b, u), s in zip(ctxs, streams):
        b.close()
        for _ in range(3):
            a.step(2)
        alone.append(a.get_moments(torch.empty_like(u)))
        a.synchronize()
        a.set_moments(u)
        a.synchronize()
        a.set_stream(s)
    torch.cuda.synchronize()
    for _ in range(3):
        for a, _, _ in ctxs:
            a.step(2)
    for (a, _, u), s, ref in zip(ctxs, streams, alone):
        a.synchronize()
        got = torch.empty_like(u)
        with torch.cuda.stream(s):
            a.get_moments(got)
        s.synchronize()
        assert torch.equal(got, ref)
        a.close()
