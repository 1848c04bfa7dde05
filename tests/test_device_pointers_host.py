"""Moments in and out through device pointers that the context's kernels may not dereference: memory of
another GPU and addresses off the type's alignment go through the runtime's copies, as page-locked
host memory does.  With a stand-in for the CUDA runtime, which shows what would be launched."""
import pytest

import fake_runtime

SCRIPT = """
N, shape, nc = {N}, {shape}, ({N} + 1) ** 2
ctx = rtpn.Context(N, shape, 0.1, "periodic", {precision!r})
padded = ctx.info().state_bytes != nc * shape[0] * shape[1] * shape[2] * {elem}
assert padded == {padded}
V = shape[0] * shape[1] * shape[2]
size = nc * V * 8 + 64
lib = rtpn.lib()
far = fake.fake_remote(size)
array = np.zeros(size, np.uint8)
host = array.ctypes.data
own = ctypes.c_void_p()
assert fake.cudaMalloc(ctypes.byref(own), ctypes.c_size_t(size)) == 0
for call in (lib.rtpn_set_moments, lib.rtpn_get_moments):
    for dtype in (0, 1):
        # the context's own GPU, aligned: one kernel, no copy
        log()
        assert call(ctx._p, own.value, dtype, 1) == 0
        seen = log()
        assert len(seen) == 1 and seen[0].startswith("K "), seen
        # another GPU, host memory, an address off the alignment: never given to a kernel over all components
        for p in (far, host, own.value + 2):
            assert call(ctx._p, p, dtype, 1) == 0
            seen = log()
            assert kernels(seen, "k_reorder") == 0, seen
            assert sum(l.startswith("C cudaMemcpyAsync") for l in seen) == nc, seen
            same = {precision!r} == ("fp64", "fp32")[dtype]
            assert sum(l.startswith("K ") for l in seen) == (0 if same and not padded else nc), seen
for call in (lib.rtpn_set_component, lib.rtpn_get_component):
    for p in (far, own.value + 2):
        assert call(ctx._p, 3, p, 1, 1) == 0
        assert sum(l.startswith("C cudaMemcpyAsync") for l in log()) == 1
"""


@pytest.fixture(scope="module")
def so(tmp_path_factory, rtpn_lib):
    return fake_runtime.build(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("N,shape,precision,elem,padded", [
    (3, (2, 3, 8), "fp32", 4, False), (3, (2, 3, 7), "fp64", 8, False), (3, (2, 3, 8), "bf16", 2, False),
    (15, (2, 3, 75), "fp32", 4, True), (15, (2, 3, 75), "bf16", 2, True)])
def test_pointers_the_kernels_may_not_read(so, N, shape, precision, elem, padded):
    fake_runtime.run(so, SCRIPT.format(N=N, shape=shape, precision=precision, elem=elem, padded=padded))
