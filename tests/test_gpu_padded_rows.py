"""Grids whose rows are no 16-byte groups: the automatic choice runs the staged kernel on padded rows.  The
step against the oracle, every way in and out of the state, moving between kernels (dense and padded
rows), plane copies between the two layouts, the diagnostics and the adjoint."""
import numpy as np
import pytest
import torch

from paper_2004_02833_gb300 import rtpn, synth
from test_gpu_parity import assert_parity, oracle_problem

pytestmark = pytest.mark.gpu

CASES = [
    # N, shape (nz, ny, nx), bc
    (15, (5, 6, 75), "periodic"),
    (15, (4, 3, 9), "vacuum"),
    (15, (3, 4, 66), "vacuum"),
    (19, (4, 5, 35), "periodic"),
    (29, (3, 2, 9), "vacuum"),
    (39, (3, 4, 81), "periodic"),
]


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("N,shape,bc", CASES)
def test_step_on_padded_rows(cuda_device, coupling_cache, N, shape, bc, precision):
    inst, u0 = synth.random_instance(N, shape, seed=1300 + N, bc=bc)
    P = oracle_problem(inst, coupling_cache)
    ref = P.run(u0, 2)
    with rtpn.Context(N, shape, inst.h, bc, precision, inst.dt) as ctx:
        assert ctx.info().kernel == 3
        with pytest.raises(rtpn.RtpnError):
            ctx.set_kernel("stage")  # by name it takes 16-byte rows only
        assert ctx.info().kernel == 3
        ctx.set_media(inst.sigma_a, inst.sigma_s, inst.q)
        ctx.set_moments(u0)
        ctx.step(2)
        ctx.synchronize()
        got = ctx.get_moments()
        assert ctx.count_nonfinite() == 0
        assert abs(ctx.sum_u0() - got[0].sum()) <= 1e-12 * np.abs(got[0]).sum()
        w = np.random.default_rng(3).standard_normal(shape)
        assert abs(ctx.detector(w) - (w * got[0]).sum()) <= 1e-12 * np.abs(w * got[0]).sum()
    assert_parity(got, ref, precision, P, u0, 2)


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_moments_through_every_call(cuda_device, precision, dtype):
    N, shape, nc = 15, (3, 4, 13), 256
    g = torch.Generator(device="cuda").manual_seed(9)
    u = torch.randn((nc,) + shape, generator=g, dtype=torch.float32, device="cuda").to(torch.bfloat16).to(dtype)
    with rtpn.Context(N, shape, 0.1, "periodic", precision) as a, rtpn.Context(N, shape, 0.1, "periodic", precision) as b:
        assert a.info().kernel == 3
        a.set_moments(u)                       # device
        b.set_moments(u.cpu())                 # host
        out = torch.empty_like(u)
        for ctx in (a, b):
            assert torch.equal(ctx.get_moments(out).clone(), u)
            assert np.array_equal(ctx.get_moments(), u.cpu().numpy().astype(np.float64))
            one = torch.empty(shape, dtype=dtype, device="cuda")
            for c in (0, 17, nc - 1):
                ctx.get_component(c, one)
                torch.cuda.synchronize()
                assert torch.equal(one, u[c])
                assert np.array_equal(ctx.get_component(c), u[c].cpu().numpy().astype(np.float64))
        # dense and padded rows and back keep every value
        for kernel in ("window", "auto", "generic", "auto"):
            a.set_kernel(kernel)
            assert a.info().kernel == {"window": 2, "auto": 3, "generic": 1}[kernel]
            assert torch.equal(a.get_moments(out).clone(), u)
        # planes between a padded and a dense state, both ways
        b.set_kernel("window")
        b.zero_moments()
        b.copy_planes_from(a, 1, 0, 2)
        ref = torch.zeros_like(u)
        ref[:, 0:2] = u[:, 1:3]
        assert torch.equal(b.get_moments(out).clone(), ref)
        a.copy_planes_from(b, 0, 2, 1, cls=-1)
        ref = u.clone()
        ref[:, 2] = u[:, 1]
        assert torch.equal(a.get_moments(out).clone(), ref)
        a.zero_moments()
        assert a.sum_u0() == 0.0


def test_kernels_agree_between_steps(cuda_device, coupling_cache):
    inst, u0 = synth.random_instance(15, (5, 4, 21), seed=1401, bc="vacuum")
    P = oracle_problem(inst, coupling_cache)
    ref = P.run(u0, 4)
    with rtpn.Context(15, inst.shape, inst.h, inst.bc, "fp32", inst.dt) as ctx:
        ctx.set_media(inst.sigma_a, inst.sigma_s, inst.q)
        ctx.set_moments(u0)
        for kernel in ("auto", "window", "auto", "generic"):
            ctx.set_kernel(kernel)
            ctx.step(1)
        assert_parity(ctx.get_moments(), ref, "fp32", P, u0, 4)
        ctx.set_kernel("auto")
        tile, ms = ctx.autotune(reps=1)
        assert ctx.info().kernel == 3 and ms > 0
        assert_parity(ctx.get_moments(), ref, "fp32", P, u0, 4)


def test_adjoint_on_padded_rows(cuda_device):
    # the adjoint runs on dense rows: the gradients of an explicit window context, and the state after it
    inst, u0 = synth.random_instance(15, (4, 5, 13), seed=1402, bc="vacuum")
    w = np.random.default_rng(4).standard_normal(inst.shape)
    res = []
    for kernel in ("auto", "window"):
        with rtpn.Context(15, inst.shape, inst.h, inst.bc, "fp32", inst.dt) as ctx:
            ctx.set_kernel(kernel)
            ctx.set_media(inst.sigma_a, inst.sigma_s, inst.q)
            ctx.set_moments(u0)
            J, g = ctx.adjoint(w, 4, ckpt_every=2)
            assert ctx.info().kernel == {"auto": 3, "window": 2}[kernel]
            res.append((J, *g, ctx.get_moments()))
    assert res[0][0] == res[1][0]
    for a, b in zip(res[0][1:], res[1][1:]):
        assert np.array_equal(a, b)
