"""Kernels that may start before the one ahead of them has ended (launch_pdl) and the read-only load path do not
go together: what an earlier kernel may still write is read by ordinary loads.  Checked on the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2004_02833_gb300", "csrc")
FIXED = {"perm"}  # written at creation only
READ_ONLY = re.compile(r"__ldg\s*\(|\bld\.global\.nc\b|\bro\s*\(|\bload_nc\b|\bload_as\b|\bsubstep_cell\b")


def sources():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh", ".h")):
            yield f, open(os.path.join(CSRC, f)).read()


def kernel(name):
    """(parameters, body) of a __global__ function."""
    for _, text in sources():
        m = re.search(r"__global__[^;{]*\b" + name + r"\s*\(([^)]*)\)\s*\{", text)
        if m:
            depth, i = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                i += 1
            return m.group(1), text[m.end():i]
    raise AssertionError(name)


def test_early_started_kernels_read_by_ordinary_loads():
    started = set()
    for _, text in sources():
        started |= set(re.findall(r"launch_pdl\(\s*(\w+)\s*<", text)) | set(re.findall(r"launch_pdl\(\s*(k_\w+)\s*,", text))
    assert started  # the moments in and out
    for name in sorted(started):
        params, body = kernel(name)
        for p in params.split(","):
            if "const" in p and "__restrict__" in p:
                assert p.split()[-1] in FIXED, (name, p)
        assert not READ_ONLY.search(body), name
        # every thread waits before anything else
        first = [s.strip() for s in body.split(";")][:2]
        assert "pdl_wait()" in first, (name, first)
