"""Runs a script against the built library with a stand-in for the CUDA runtime preloaded (no GPU): see
tests/host/fake_cudart.cpp."""
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
_exe = {}

HEAD = """
import collections, ctypes, sys
import numpy as np
sys.path.insert(0, {root!r})
fake = ctypes.CDLL({so!r})
fake.fake_log.restype = ctypes.c_char_p
fake.fake_remote.restype = ctypes.c_void_p
fake.fake_remote.argtypes = [ctypes.c_size_t]
fake.fake_limit.argtypes = [ctypes.c_size_t]
fake.fake_used.restype = ctypes.c_size_t
from paper_2004_02833_gb300 import rtpn

def fail(api, after=0, code=1):
    fake.fake_fail(api.encode(), after, code)

def log():
    lines = [l for l in fake.fake_log().decode().split("\\n") if l]
    fake.fake_clear()
    return lines

def kernels(lines, name):
    return sum(l.startswith("K ") and name in l for l in lines)

def code(fn, *a):
    try:
        fn(*a)
    except rtpn.RtpnError as e:
        return e.code
    return rtpn.OK
"""


def build(tmp):
    cuda = "/usr/local/cuda/include"
    if shutil.which("g++") is None or not os.path.isdir(cuda):
        pytest.skip("g++ or the CUDA headers are not available")
    so = os.path.join(str(tmp), "fake_cudart.so")
    res = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + cuda,
                          os.path.join(HERE, "host", "fake_cudart.cpp"), "-o", so], capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]
    return so


def run(so, script, env=None):
    """Runs the script after HEAD; it has to end with status 0 (its asserts are the test)."""
    src = HEAD.format(root=ROOT, so=so) + textwrap.dedent(script)
    e = dict(os.environ, LD_PRELOAD=so, **(env or {}))
    res = subprocess.run([sys.executable, "-c", src], capture_output=True, text=True, timeout=300, env=e)
    assert res.returncode == 0, res.stdout[-1000:] + res.stderr[-3000:]
    return res.stdout
