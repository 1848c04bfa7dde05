"""What users of this framework have it do, as cases that can be timed: time stepping of the P_N moment
system at the orders, grids, storage types and options of the benchmark and the tests, the training
step through the adjoint, and the batched form.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (a context with
its media and state, buffers for the results), ``run`` is the call, ``exact`` the same result from a
plain 64-bit restatement of the method (quadrature coupling matrices, whole-array shifts).
"""
import math

import numpy as np
import torch

from paper_2004_02833_gb300 import autograd, rtpn

ORDERS = (1, 3, 5, 7, 9, 15, 19, 29, 39)  # orders of the benchmark, the showcase and the tests
BATCH_ORDERS = (1, 3, 5, 9, 15)           # of the batched benchmark
H = 0.1                                   # cell size (the method only sees dt/h and sigma*dt)


def _step(name, N, shape, steps, bc="periodic", precision="fp32", media="blocks", spacing=False, aniso=False):
    nz, ny, nx = shape
    return {"name": name, "kind": "step", "N": N, "nz": nz, "ny": ny, "nx": nx, "steps": steps, "bc": bc,
            "precision": precision, "media": media, "spacing": spacing, "aniso": aniso}


def listed():
    return [
        # an interactive or coupled loop that advances a small pulse problem one step at a time and
        # reads the moments after each: launches and copies are all there is
        _step("p3_32_one_step", 3, (32, 32, 32), 1, media="uniform"),
        # the plain pulse problem in the reference precision, as a convergence check runs it
        _step("p3_32_fp64", 3, (32, 32, 32), 40, precision="fp64", media="uniform"),
        # the lattice (checkerboard) problem at its usual size
        _step("p7_128_lattice", 7, (128, 128, 128), 10, bc="vacuum", media="lattice"),
        # a box with odd extents and cells that are not cubes
        _step("p7_ragged_box", 7, (67, 90, 101), 10, spacing=True),
        # anisotropic (Henyey-Greenstein) scattering
        _step("p7_96_aniso", 7, (96, 96, 96), 10, aniso=True),
        # the high orders of a convergence study on a grid whose rows are not 16-byte multiples
        _step("p15_ragged", 15, (61, 77, 75), 5),
        # the lattice problem at the order of the adjoint benchmark
        _step("p15_96_lattice", 15, (96, 96, 96), 5, bc="vacuum", media="lattice"),
        # the order that resolves the reactor showcase
        _step("p19_80_lattice", 19, (80, 80, 80), 3, bc="vacuum", media="lattice"),
        # the headline problem's order and media, on a grid three states of which fit the card
        _step("p39_160_blocks", 39, (160, 160, 160), 2),
        # the same with BF16 storage
        _step("p39_120_bf16", 39, (120, 120, 120), 4, precision="bf16"),
        # one training iteration over the media: forward, detector, discrete adjoint
        {"name": "adjoint_p15_64", "kind": "adjoint", "N": 15, "nz": 64, "ny": 64, "nx": 64, "steps": 20,
         "every": 10, "bc": "vacuum"},
        # many uneven instances advanced together
        {"name": "batch_24", "kind": "batch", "count": 24, "lo": 24, "hi": 96, "steps": 4, "shapes": 3},
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step",) * 6 + ("adjoint", "batch"))
    if kind == "batch":
        lo = rng.randint(16, 40)
        return {"kind": "batch", "count": rng.randint(4, 24), "lo": lo, "hi": rng.randint(lo + 8, 96),
                "steps": rng.randint(2, 6), "shapes": rng.randint(0, 1 << 20)}
    if kind == "adjoint":
        # the orders whose FP32 adjoint a user trains with; rows in multiples of four cells
        steps = rng.randint(4, 20)
        return {"kind": "adjoint", "N": rng.choice((7, 15)), "nz": _side(rng, 16, 64), "ny": _side(rng, 16, 64),
                "nx": 4 * _side(rng, 4, 16), "steps": steps, "every": rng.randint(2, max(2, steps // 2)),
                "bc": rng.choice(("periodic", "vacuum"))}
    N = rng.choice(ORDERS)
    precision = "fp64" if N <= 9 and rng.random() < 0.15 else "bf16" if rng.random() < 0.25 else "fp32"
    top = {1: 200, 3: 192, 5: 160, 7: 144, 9: 128, 15: 112, 19: 96, 29: 96, 39: 112}[N]
    if precision == "fp64":
        top = 64
    nz, ny, nx = (_side(rng, 20, top) for _ in range(3))
    if rng.random() < 0.7:
        nx = max(16, nx // 8 * 8)  # most users take round widths
    bc = rng.choice(("periodic", "vacuum"))
    option = rng.choice(("", "", "spacing", "aniso")) if N <= 15 else ""
    c = _step("", N, (nz, ny, nx), rng.randint(1, 12), bc, precision, rng.choice(("blocks", "lattice", "uniform")),
              option == "spacing", option == "aniso")
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _media(kind, shape, seed):
    """sigma_a, sigma_s, q, float64 on the GPU: a homogeneous scatterer, random 8^3 blocks, or the
    7^3-block lattice of absorbers and scatterers with a source in its centre."""
    g = _generator(seed)
    axis = [torch.arange(n, device="cuda") for n in shape]
    if kind == "lattice":
        b = [torch.clamp((a * 7) // n, max=6) for a, n in zip(axis, shape)]
        Z, Y, X = torch.meshgrid(*b, indexing="ij")
        inner = (X >= 1) & (X <= 5) & (Y >= 1) & (Y <= 5) & (Z >= 1) & (Z <= 5)
        centre = (X == 3) & (Y == 3) & (Z == 3)
        absorber = inner & ((X + Y + Z) % 2 == 1) & ~centre
        scale = 0.9 + 0.2 * torch.rand((7, 7, 7), generator=g, dtype=torch.float64, device="cuda")[Z, Y, X]
        zero = torch.zeros_like(scale)
        return (torch.where(absorber, 10.0 * scale, zero), torch.where(absorber, zero, scale),
                torch.where(centre, scale, zero))
    if kind == "blocks":
        nb = [-(-n // 8) for n in shape]
        vals = torch.exp(math.log(0.1) + math.log(100.0) * torch.rand(nb, generator=g, dtype=torch.float64, device="cuda"))
        i = [a // 8 for a in axis]
        ss = vals[i[0]][:, i[1]][:, :, i[2]].contiguous()
    else:
        ss = torch.full(shape, 0.5, dtype=torch.float64, device="cuda") + torch.rand(1, generator=g, dtype=torch.float64, device="cuda")
    return torch.full_like(ss, 0.01), ss, torch.zeros_like(ss)


def _fill_state(out, seed, bf16=False):
    """A state as it stands amid a run: every moment nonzero, falling off with its order l."""
    g = _generator(seed + 1)
    for c in range(out.shape[0]):
        out[c].normal_(generator=g).mul_(1.0 / (1 + math.isqrt(c)) ** 2)
    if bf16:  # values that the storage holds as they are
        for c in range(out.shape[0]):
            out[c].copy_(out[c].to(torch.bfloat16))
    return out


def _spacing(case):
    return (H, 1.3 * H, 1.7 * H) if case.get("spacing") else (H, H, H)


def _profile(case):
    return [0.8 ** l for l in range(case["N"] + 1)] if case.get("aniso") else None


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _instances(case):
    """The batch's uneven instances: order, shape, boundary and media, by the rules of the batched benchmark."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["count"]):
        N, n = int(rng.choice(BATCH_ORDERS)), int(rng.integers(case["lo"], case["hi"] + 1))
        pulse = bool(rng.integers(0, 2))
        out.append((N, (n, n, n), "periodic" if pulse else "vacuum", "uniform" if pulse else "lattice"))
    return out


def _detector(shape):
    """Weights of a box of cells off the centre."""
    w = torch.zeros(shape, dtype=torch.float64, device="cuda")
    z, y, x = shape[0] * 7 // 16, shape[1] * 7 // 16, shape[2] * 3 // 4
    w[z:z + max(1, shape[0] // 8), y:y + max(1, shape[1] // 8), x:x + max(1, shape[2] // 8)] = 1.0
    return w


def prepare(case, seed):
    if case["kind"] == "batch":
        inst = _instances(case)
        batch = rtpn.Batch([(N, shape, H, bc, None) for N, shape, bc, _ in inst])
        outs = []
        for i, (N, shape, bc, media) in enumerate(inst):
            out = torch.empty(((N + 1) ** 2,) + shape, dtype=torch.float32, device="cuda")
            batch[i].set_media(*_media(media, shape, seed + 100 * i))
            batch[i].set_moments(_fill_state(out, seed + 100 * i))
            batch[i].synchronize()
            outs.append(out)
        return {"case": case, "batch": batch, "outs": outs}
    shape, N = _shape(case), case["N"]
    if case["kind"] == "adjoint":
        media = _media("lattice", shape, seed)
        u = _fill_state(torch.empty(((N + 1) ** 2,) + shape, dtype=torch.float32, device="cuda"), seed)
        ctx = rtpn.Context(N, shape, H, bc=case["bc"], precision="fp32")
        return {"case": case, "ctx": ctx, "media": [m.requires_grad_() for m in media], "u": u, "w": _detector(shape)}
    ctx = rtpn.Context(N, shape, H, bc=case["bc"], precision=case["precision"])
    if case["spacing"]:
        ctx.set_spacing(*_spacing(case))
    if case["aniso"]:
        ctx.set_scattering(_profile(case))
    out = torch.empty(((N + 1) ** 2,) + shape, dtype=_dtype(case), device="cuda")
    ctx.set_media(*_media(case["media"], shape, seed))
    ctx.set_moments(_fill_state(out, seed, case["precision"] == "bf16"))
    ctx.synchronize()
    return {"case": case, "ctx": ctx, "out": out}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        return [state["batch"][i].get_moments(out) for i, out in enumerate(state["outs"])]
    if case["kind"] == "adjoint":
        sa, ss, q = state["media"]
        J = autograd.detector_response(state["ctx"], sa, ss, q, state["u"], state["w"], case["steps"], case["every"])
        return [J.detach(), *torch.autograd.grad(J, (sa, ss, q))]
    state["ctx"].step(case["steps"])
    out = state["ctx"].get_moments(state["out"])
    # a BF16 state is kept as BF16 (the same values: they come from that storage)
    return out.to(torch.bfloat16) if case["precision"] == "bf16" else out


# ---------------------------------------------------------------- what a pass cannot do without
def _counts(N):
    """Components, and their nonzero couplings over the three axes."""
    n = nz = 0
    for l in range(N + 1):
        for m in range(-l, l + 1):
            n += 1
            nz += len(_partners(N, l, m))
    return n, nz


def _valid(N, l, m):
    return 0 <= l <= N and -l <= m <= l


def _partners(N, l, m):
    """(axis, l', m') that the three direction cosines couple (l, m) to."""
    M, sign = abs(m), -1 if m < 0 else 1
    out = [(2, l + d, m) for d in (-1, 1)]
    for d in (-1, 1):
        for Mt in (M - 1, M + 1):
            if Mt < 0:
                continue
            same, other = sign * Mt, -sign * Mt
            if Mt > 0 or sign > 0:
                out.append((0, l + d, same))
            if M == 0:
                out.append((1, l + d, -Mt))
            elif Mt > 0:
                out.append((1, l + d, other))
            elif sign < 0:
                out.append((1, l + d, 0))
    return [(a, lp, mp) for a, lp, mp in out if _valid(N, lp, mp)]


def _one_run(N, cells, steps, elem):
    """State in and out once a step with the media's factors of each cell, and the flops of Eq. (5)."""
    n, nz = _counts(N)
    return steps * cells * (2.0 * n * elem + 12.0), steps * cells * (2.0 * nz + 3.0 * n + 4.0 * n)


def work(case):
    if case["kind"] == "batch":
        b = f = 0.0
        for N, shape, _, _ in _instances(case):
            cells = float(np.prod(shape))
            x, y = _one_run(N, cells, case["steps"], 4)
            b, f = b + x + cells * (N + 1) ** 2 * 8.0, f + y
        return {"bytes": b, "flops": f}
    N, cells = case["N"], float(np.prod(_shape(case)))
    n = (N + 1) ** 2
    if case["kind"] == "adjoint":
        # the forward, its states kept, and a backward of the same traffic; media and gradients
        x, y = _one_run(N, cells, case["steps"], 4)
        return {"bytes": 2.5 * x + cells * (n * 4.0 + 56.0), "flops": 2.0 * y}
    elem = {"fp64": 8, "fp32": 4, "bf16": 2}[case["precision"]]
    x, y = _one_run(N, cells, case["steps"], elem)
    return {"bytes": x + 2.0 * cells * n * elem, "flops": y}


# ---------------------------------------------------------------- the method in 64 bits
def _basis(N, mu, phi):
    """Real orthonormal spherical harmonics, no Condon-Shortley phase, rows c = l*l + l + m."""
    s = np.sqrt(1.0 - mu * mu)
    Y = np.zeros(((N + 1) ** 2, mu.size))
    pmm = np.full_like(mu, math.sqrt(1.0 / (4.0 * math.pi)))
    for M in range(N + 1):
        if M > 0:
            pmm = pmm * s * math.sqrt((2 * M + 1) / (2.0 * M))
        lo, cur = np.zeros_like(mu), pmm
        for l in range(M, N + 1):
            if M == 0:
                Y[l * l + l] = cur
            else:
                Y[l * l + l + M] = math.sqrt(2.0) * cur * np.cos(M * phi)
                Y[l * l + l - M] = math.sqrt(2.0) * cur * np.sin(M * phi)
            a = math.sqrt((4.0 * (l + 1) ** 2 - 1) / ((l + 1) ** 2 - M * M))
            b = math.sqrt((l * l - M * M) / (4.0 * l * l - 1)) if l > 0 else 0.0
            lo, cur = cur, a * (mu * cur - b * lo)
    return Y


def _matrices(N):
    """Mx, My, Mz by a product rule that is exact for them, and each component's slots (x, y, z)."""
    x, wx = np.polynomial.legendre.leggauss(N + 4)
    n_phi = 2 * N + 8
    mu, phi = (a.ravel() for a in np.meshgrid(x, 2 * math.pi * np.arange(n_phi) / n_phi, indexing="ij"))
    w = np.repeat(wx, n_phi) * (2 * math.pi / n_phi)
    Y, s = _basis(N, mu, phi), np.sqrt(1 - mu * mu)
    mats = [(Y * (w * o)) @ Y.T for o in (s * np.cos(phi), s * np.sin(phi), mu)]
    for m in mats:
        m[np.abs(m) < 1e-10] = 0.0
    slots = []
    for l in range(N + 1):
        for m in range(-l, l + 1):
            even = abs(m) % 2 == 0
            slots.append((1 if even == (m >= 0) else 2, 1 if m >= 0 else 2, 1 if (l + m) % 2 == 0 else 2))
    return mats, slots


def _shift(f, axis, s, periodic):
    """f(i + s e_axis), axis 0 x, 1 y, 2 z, over the last three dimensions; zero outside a vacuum box."""
    dim = -1 - axis
    g = torch.roll(f, -s, dim)
    if not periodic:
        n = f.shape[dim]
        g.narrow(dim, n - 1 if s > 0 else 0, 1).zero_()
    return g


def _point_mean(f, slot, periodic):
    tot, cnt = f, torch.ones_like(f)
    for d in range(3):
        if slot[d] == 2:
            tot, cnt = tot + _shift(tot, d, 1, periodic), cnt + _shift(cnt, d, 1, periodic)
    return tot / cnt


def _factors(c, tau):
    """exp(-c tau) and (1 - exp(-c tau)) / c, tau - c tau^2 / 2 where c is 0."""
    safe = torch.where(c == 0, torch.ones_like(c), c)
    return torch.exp(-c * tau), torch.where(c == 0, tau - 0.5 * tau * tau * c, -torch.expm1(-safe * tau) / safe)


class _Method:
    """Eq. (3)-(6) on whole arrays in float64."""

    def __init__(self, N, media, bc, spacing=(H, H, H), profile=None):
        self.N, self.periodic, self.h, self.profile = N, bc == "periodic", spacing, profile
        self.sa, self.ss, self.q = media
        self.mats, self.slots = _matrices(N)
        self.dt = 0.3 * spacing[0]
        self.cls = [sum(g == 2 for g in s) % 2 for s in self.slots]
        self.cache = {}

    def factors(self, a, tau):
        l = math.isqrt(a)
        key = (self.slots[a], tau, 0 if a == 0 else 1, l if self.profile else 0)
        if key not in self.cache:
            total = self.sa if a == 0 else self.sa + (1.0 - self.profile[l]) * self.ss if self.profile else self.sa + self.ss
            self.cache[key] = _factors(_point_mean(total, self.slots[a], self.periodic), tau)
        return self.cache[key]

    def difference(self, u, d, target_slot):
        if target_slot == 2:
            return _shift(u, d, 1, self.periodic) - u
        return u - _shift(u, d, -1, self.periodic)

    def substep(self, u, cls, tau):
        """In place: every component of the class, the other class frozen."""
        for a in range(len(self.slots)):
            if self.cls[a] != cls:
                continue
            r = self.q.clone() if a == 0 else torch.zeros_like(self.q)
            for d in range(3):
                for b in np.nonzero(self.mats[d][a])[0]:
                    r.add_(self.difference(u[b], d, self.slots[a][d]), alpha=-float(self.mats[d][a, b]) / self.h[d])
            al, be = self.factors(a, tau)
            u[a].mul_(al).addcmul_(be, r)

    def steps(self, u, k):
        for _ in range(k):
            self.substep(u, 1, 0.5 * self.dt)
            self.substep(u, 0, self.dt)
            self.substep(u, 1, 0.5 * self.dt)
        return u

    def differentiable(self, u, k):
        """The same by matrix products over the classes, for autograd."""
        idx = [[a for a in range(len(self.slots)) if self.cls[a] == c] for c in (0, 1)]
        parts = [u[i] for i in idx]
        fac = {}
        for cls, tau in ((1, 0.5 * self.dt), (0, self.dt)):
            f = [self.factors(a, tau) for a in idx[cls]]
            fac[cls] = (torch.stack([x[0] for x in f]), torch.stack([x[1] for x in f]))
        blocks = {(c, d): torch.tensor(self.mats[d][np.ix_(idx[c], idx[1 - c])] / self.h[d], device=u.device)
                  for c in (0, 1) for d in range(3)}

        def advance(cls):
            src, r = parts[1 - cls], 0.0
            for d in range(3):
                # a source on slot 1 is read at i and i + 1 by its partners on slot 2, and the other way round
                up = torch.tensor([self.slots[b][d] == 1 for b in idx[1 - cls]], device=u.device).view(-1, 1, 1, 1)
                D = torch.where(up, _shift(src, d, 1, self.periodic) - src, src - _shift(src, d, -1, self.periodic))
                r = r - torch.tensordot(blocks[cls, d], D, dims=([1], [0]))
            if cls == 0:
                r = torch.cat([r[:1] + self.q, r[1:]])
            parts[cls] = fac[cls][0] * parts[cls] + fac[cls][1] * r

        for _ in range(k):
            for cls in (1, 0, 1):
                advance(cls)
        return parts[0][0]


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "batch":
            outs = []
            for i, (N, shape, bc, media) in enumerate(_instances(case)):
                u = _fill_state(torch.empty(((N + 1) ** 2,) + shape, dtype=torch.float32, device="cuda"), seed + 100 * i)
                outs.append(_Method(N, _media(media, shape, seed + 100 * i), bc).steps(u.double(), case["steps"]))
            return outs
        shape, N = _shape(case), case["N"]
        if case["kind"] == "step":
            u = _fill_state(torch.empty(((N + 1) ** 2,) + shape, dtype=_dtype(case), device="cuda"), seed,
                            case["precision"] == "bf16")
            u = u if u.dtype == torch.float64 else u.double()
            m = _Method(N, _media(case["media"], shape, seed), case["bc"], _spacing(case), _profile(case))
            return m.steps(u, case["steps"])
    cells = float(np.prod(shape))
    if (N + 1) ** 2 * cells * case["steps"] > 2.0e9:
        return None  # the graph of the differentiated steps takes too long
    media = [x.requires_grad_() for x in _media("lattice", shape, seed)]
    u = _fill_state(torch.empty(((N + 1) ** 2,) + shape, dtype=torch.float32, device="cuda"), seed)
    m = _Method(N, media, case["bc"])
    J = (m.differentiable(u.double(), case["steps"]) * _detector(shape)).sum()
    return [J.detach(), *torch.autograd.grad(J, media)]
