"""Kernel selection, row pitch and allocation against failures of the calls they make, with a stand-in for the
CUDA runtime (no GPU): whatever fails, the kernel in use and the rows of the state go together, and the
error is reported."""
import pytest

import fake_runtime


@pytest.fixture(scope="module")
def so(tmp_path_factory, rtpn_lib):
    return fake_runtime.build(tmp_path_factory.mktemp("fake"))


COMMON = """
shape = (3, 4, 75)
V = 3 * 4 * 75
dense, padded = 256 * V * 4, 256 * 3 * 4 * 76 * 4
def layout(ctx):
    i = ctx.info()
    return i.kernel, i.state_bytes
def fits(ctx):
    return layout(ctx) in ((1, dense), (2, dense), (3, padded))
def context(media=True):
    ctx = rtpn.Context(15, shape, 0.1)
    assert layout(ctx) == (3, padded)
    if media:
        m = np.full(shape, 0.5)
        ctx.set_media(m, m, m)
    log()
    return ctx
"""


def test_a_failed_selection_leaves_kernel_and_rows(so):
    fake_runtime.run(so, COMMON + """
ctx = context()
tile = tuple(ctx.info().tile)
ctx.set_kernel("window", (32, 4, 1))
for api, after in (("cudaMemcpy", 0),):
    fail(api, after, 719)
    log()
    assert code(ctx.set_kernel, "auto") == rtpn.ECUDA
    assert layout(ctx) == (2, dense) and tuple(ctx.info().tile) == (32, 4, 1)
    assert kernels(log(), "k_rows") == 0  # the state was not touched
ctx.set_kernel("auto")
assert layout(ctx) == (3, padded) and tuple(ctx.info().tile) == tile
# from the staged kernel to one that cannot be had: the staged kernel and its rows stay
log()
assert code(ctx.set_kernel, "fused") == rtpn.EUNSUPPORTED
assert layout(ctx) == (3, padded) and tuple(ctx.info().tile) == tile
assert kernels(log(), "k_rows") == 0
""")


def test_set_up_that_fails_for_want_of_memory(so):
    fake_runtime.run(so, COMMON + """
ctx = context()
ctx.set_kernel("window")
ctx.set_spacing(0.1, 0.1, 0.1)  # drops the staged kernel's tables
fail("cudaMalloc", 0, 2)
log()
assert code(ctx.set_kernel, "auto") != rtpn.OK
assert layout(ctx) == (2, dense)
assert kernels(log(), "k_rows") == 0
ctx.set_kernel("auto")
assert layout(ctx) == (3, padded)
""")


def test_adjoint_on_padded_rows_returns_what_its_way_back_met(so):
    fake_runtime.run(so, COMMON + """
ctx = context()
w = np.ones(shape)
ctx.adjoint(w, 2, ckpt_every=2)
assert layout(ctx) == (3, padded)
lines = log()
# the way back to padded rows is queued before the last wait, so that its errors are the call's
rows = max(i for i, l in enumerate(lines) if l.startswith("K ") and "k_rows" in l)
assert rows < max(i for i, l in enumerate(lines) if l == "S")
copies = sum(l.startswith("C cudaMemcpy ") for l in lines)
assert copies > 0
# the last of them sets up the staged kernel again
fail("cudaMemcpy", copies - 1, 719)
assert code(ctx.adjoint, w, 2, 2) == rtpn.ECUDA
assert fits(ctx), layout(ctx)
ctx.set_kernel("auto")
ctx.step(1)
assert fits(ctx)
# an error inside: reported as itself, with the rows padded again
ctx = context()
fail("cudaMalloc", 2, 2)
assert code(ctx.adjoint, w, 2, 2) == rtpn.ENOMEM
assert layout(ctx) == (3, padded)
""")


def test_auto_with_a_depth_on_rows_that_are_no_16_byte_groups(so):
    # a depth that a variant has runs staged; one that none has leaves the kernels that take any width
    fake_runtime.run(so, """
for precision in ("fp32", "bf16"):
    for N, any_width in ((15, 2), (19, 1), (29, 1), (39, 2)):
        ctx = rtpn.Context(N, (2, 3, 75), 0.1, "periodic", precision)
        assert ctx.info().kernel == 3
        for depth in range(9):
            assert code(ctx.set_kernel, "auto", (0, 0, 0), depth) == rtpn.OK, (N, depth)
            i = ctx.info()
            assert i.kernel in (3, any_width) and (i.kernel != 3 or depth in (0, i.depth)), (N, depth)
            dense = (N + 1) ** 2 * 2 * 3 * 75 * (4 if precision == "fp32" else 2)
            assert (i.state_bytes != dense) == (i.kernel == 3)
        # on 16-byte rows such a depth is refused, as by name, and the selection stays
        even = rtpn.Context(N, (2, 3, 72), 0.1, "periodic", precision)
        assert code(even.set_kernel, "auto", (0, 0, 0), 8) == rtpn.EUNSUPPORTED
        assert even.info().kernel == 3
""")


def test_padding_is_not_what_keeps_a_problem_off_the_device(so):
    # nx = 9 in BF16 pads to 16: the state alone needs 16/9 of the dense one
    fake_runtime.run(so, """
shape = (40, 40, 9)
def used(kernel):
    ctx = rtpn.Context(15, shape, 0.1, "periodic", "bf16")
    if kernel:
        ctx.set_kernel(kernel)
    b = fake.fake_used(), ctx.info().state_bytes, ctx.info().kernel
    ctx.close()
    return b
room, padded, kernel = used(None)
dense = 256 * 40 * 40 * 9 * 2
assert kernel == 3 and padded == dense * 16 // 9 and fake.fake_used() == 0
least = room - (padded - dense)  # what the dense form of the same context takes (the tables included)
for limit in range(least, room, (padded - dense) // 7):
    fake.fake_limit(limit)
    ctx = rtpn.Context(15, shape, 0.1, "periodic", "bf16")
    assert ctx.info().kernel == 2 and ctx.info().state_bytes == dense
    m = np.full(shape, 0.5)
    ctx.set_kernel("generic")
    ctx.set_kernel("auto")
    assert ctx.info().kernel == 2 and ctx.info().state_bytes == dense
    ctx.close()
    assert fake.fake_used() == 0
fake.fake_limit(room)
assert used(None) == (room, padded, 3)
fake.fake_limit(dense)
assert code(rtpn.Context, 15, shape, 0.1, "periodic", "bf16") == rtpn.ENOMEM
assert fake.fake_used() == 0
""")


def test_tuner_on_padded_rows_tries_every_staged_tile(so):
    fake_runtime.run(so, """
import re
text = open({root!r} + "/paper_2004_02833_gb300/csrc/stage_variants.h").read()
tiles = [tuple(map(int, m)) for m in re.findall(r"X\\(15,\\s*(\\d+),\\s*(\\d+),\\s*(\\d+),\\s*(\\d+),", text)]
assert len(tiles) > 4
shape = (3, 4, 75)
m = np.full(shape, 0.5)
def use(i):
    return tuple(i.tile) + (i.depth,)
fake.fake_elapsed.argtypes = [ctypes.c_float, ctypes.c_float]
for first, step, best in ((100.0, 1.0, tiles[0]), (1000.0, -1.0, tiles[-1])):
    ctx = rtpn.Context(15, shape, 0.1, "periodic" if step > 0 else "vacuum")
    ctx.set_media(m, m, m)
    fake.fake_elapsed(first, step)
    log()
    tile, ms = ctx.autotune(reps=1)
    assert len({{l for l in log() if "k_stage" in l}}) == len(tiles) * 2  # both classes of every variant
    info = ctx.info()
    assert (info.kernel, use(info), tile) == (3, best, best[:3])
    # the adjoint's way over dense rows, and other cells, keep the tuned tile
    ctx.adjoint(m, 1, ckpt_every=1)
    assert (ctx.info().kernel, use(ctx.info())) == (3, best)
    # a second context of the same problem takes it from the tuner's memory
    other = rtpn.Context(15, shape, 0.1, "periodic" if step > 0 else "vacuum")
    other.set_media(m, m, m)
    assert other.autotune(reps=1)[0] == best[:3] and use(other.info()) == best
    # a tile that fails to be set leaves the one in use
    fail("cudaMemcpy", 0, 719)
    assert code(other.autotune, 1) == rtpn.ECUDA and use(other.info()) == best and other.info().kernel == 3
""".format(root=fake_runtime.ROOT))


def test_components_of_4_gib_are_refused_at_the_selection(so):
    # the staged kernel's byte strides are 32-bit: AUTO takes another kernel, the kernel by name is refused
    fake_runtime.run(so, """
for precision, nz in (("fp32", 1024), ("bf16", 2048)):
    for nx, kernel in ((1016, 3), (1024, 2)):
        ctx = rtpn.Context(15, (nz, 1024, nx), 0.1, "periodic", precision)
        assert ctx.info().kernel == kernel, (precision, nx)
        assert code(ctx.set_kernel, "stage") == (rtpn.OK if kernel == 3 else rtpn.EUNSUPPORTED)
        assert ctx.info().kernel == kernel
        ctx.close()
    # rows that would reach it by their padding
    ctx = rtpn.Context(15, (nz, 1024, 1023), 0.1, "periodic", precision)
    assert ctx.info().kernel == 2
    ctx.close()
""")


def test_rows_are_not_rearranged_into_the_callers_graph(so):
    fake_runtime.run(so, COMMON + """
ctx = context()
fake.fake_capturing(1)
for kernel in ("window", "generic"):
    assert code(ctx.set_kernel, kernel) == rtpn.ESTATE
    assert layout(ctx) == (3, padded) and kernels(log(), "k_rows") == 0
ctx.step(1)  # the staged passes can be captured
assert any("k_stage" in l for l in log())
fake.fake_capturing(0)
ctx.set_kernel("window")
fake.fake_capturing(1)
ctx.set_kernel("generic")  # dense rows both: nothing to rearrange
assert code(ctx.set_kernel, "auto") == rtpn.ESTATE
assert layout(ctx) == (1, dense)
""")


def test_window_passes_prefetch_where_the_data_do_not_stay_in_l2(so):
    # the default tile shows the choice: 32 x 4 x 1 with the requests to L2, 32 x 4 x 2 without (every other order too)
    fake_runtime.run(so, """
def threads(N, shape, precision, aniso=False, spacing=None):
    ctx = rtpn.Context(N, shape, 0.1, "periodic", precision)
    ctx.set_kernel("window")
    if aniso:
        ctx.set_scattering([0.8 ** l for l in range(N + 1)])
    if spacing:
        ctx.set_spacing(*spacing)
    m = np.full(shape, 0.5)
    ctx.set_media(m, m, m)
    log()
    ctx.substep(0)
    t = [int(l.split()[-1]) for l in log() if "k_window" in l]
    ctx.close()
    assert len(t) == 1
    return t[0]

for N in (5, 7, 9):
    for precision, elem in (("fp32", 4), ("bf16", 2)):
        for aniso in (False, True):
            cell = (N + 1) ** 2 * elem + 12 + (32 * (N + 1) if aniso else 64)
            nz = int(100e6 / (cell * 32 * 32))
            assert threads(N, (nz, 32, 32), precision, aniso) == 256
            assert threads(N, (nz + 1, 32, 32), precision, aniso) == 128
            assert threads(N, (8, 9, 10), precision, aniso, (0.1, 0.12, 0.13)) == 256
for N in (1, 3, 15):
    assert threads(N, (64, 64, 64), "fp32") == 256
""")


def test_default_tile_of_small_grids_at_high_orders_is_sub_staged(so):
    # columns in one stage of 15 or 20 slots are slower at any size: they run by name (or by a depth) only
    fake_runtime.run(so, """
import itertools, random, re
text = open({root!r} + "/paper_2004_02833_gb300/csrc/stage_variants.h").read()
one = {{tuple(map(int, m[:5])) for m in re.findall(r"X\\((\\d+), (\\d+), (\\d+), (\\d+), (\\d+), (\\d+)\\)", text) if m[5] == "1"}}
assert any(v[0] == 39 for v in one) and any(v[0] == 29 for v in one)
rng = random.Random(1)
for N in (29, 39):
    for precision in ("fp32", "bf16"):
        for _ in range(60):
            shape = tuple(rng.randint(1, 64) for _ in range(2)) + (rng.randint(8, 130),)
            ctx = rtpn.Context(N, shape, 0.1, "periodic", precision)
            i = ctx.info()
            assert i.kernel == 3 and (N, *i.tile, i.depth) not in one, (shape, tuple(i.tile), i.depth)
            ctx.close()
    ctx = rtpn.Context(N, (4, 4, 64), 0.1)
    for v in sorted(one):
        if v[0] == N and not (N == 39 and v[4] == 4):  # (four buffers of 40 cells fit BF16 only)
            ctx.set_kernel("stage", v[1:4], v[4])
            assert (N, *ctx.info().tile, ctx.info().depth) == v
""".format(root=fake_runtime.ROOT))


def test_pitch_of_padded_rows(so):
    # 16-byte groups; FP32 rows below 40 cells whole 32-byte sectors; 16-byte rows stay as they are
    fake_runtime.run(so, """
for precision, elem in (("fp32", 4), ("bf16", 2)):
    for N in (15, 39):
        for nx in range(1, 70):
            ctx = rtpn.Context(N, (2, 3, nx), 0.1, "periodic", precision)
            group = 16 // elem
            if nx % group == 0:
                px = nx
            elif nx < 8:
                px = nx  # not padded: a kernel that takes any width
            elif precision == "fp32" and nx < 40:
                px = -(-nx // 8) * 8
            else:
                px = -(-nx // group) * group
            i = ctx.info()
            assert i.state_bytes == (N + 1) ** 2 * 2 * 3 * px * elem, (precision, nx)
            assert (i.kernel == 3) == (px % group == 0), (precision, nx, i.kernel)
            ctx.close()
""")


def test_spacing_and_scattering_that_fail_leave_the_context(so):
    fake_runtime.run(so, COMMON + """
f = [0.8 ** l for l in range(16)]
for option in ("spacing", "scattering"):
    failed = 0
    for after in range(8):
        for api in ("cudaMalloc", "cudaMemcpy"):
            ctx = context()
            call = (lambda: ctx.set_spacing(0.1, 0.13, 0.17)) if option == "spacing" else (lambda: ctx.set_scattering(f))
            before = fake.fake_used(), layout(ctx), ctx.info().hy, ctx.info().factor_bytes, tuple(ctx.info().tile)
            fail(api, after, 2)
            rc = code(call)
            fake.fake_fail(api.encode(), 1 << 30, 0)
            if rc == rtpn.OK:
                continue
            failed += 1
            now = fake.fake_used(), layout(ctx), ctx.info().hy, ctx.info().factor_bytes, tuple(ctx.info().tile)
            assert now == before, (option, api, after, now, before)
            ctx.step(2)  # its kernels still have their tables
            assert layout(ctx) == (3, padded)
            ctx.close()
    assert failed >= 4, (option, failed)
ctx = context()
ctx.set_spacing(0.1, 0.13, 0.17)
assert ctx.info().hy == 0.13
ctx.set_spacing(0.1, 0.1, 0.1)
ctx.set_scattering(f)
assert layout(ctx) == (2, dense)
ctx.set_scattering(None)
assert layout(ctx) == (3, padded)
""")
