"""The staged kernel's ring of stage buffers when a wait runs out, on a host model of its barriers (random order
of the agents, no GPU): no producer arrives on a full barrier whose phase is not the stage's, none takes
a wait for its own copies as over while they are in flight, and no copy outlives the CTA.  The same
model with the mistake planted (consumers hand buffers back after a wait ran out) reports it."""
import os
import subprocess

import pytest

from test_fused_host import CSRC, HERE, ROOT, _nvcc

RUNS = 400


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("ring") / "model_ring")
    cmd = [nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-diag-suppress", "20011",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC, os.path.join(HERE, "host", "model_ring.cu"),
           os.path.join(CSRC, "model.cpp"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr[-2000:]

    def run(seed, skip, lp, lc, plant=False):
        r = subprocess.run([exe, str(seed), str(RUNS), str(skip), str(lp), str(lc)] + (["plant"] if plant else []),
                           capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-500:]
        return dict(zip(("rearm", "overlap", "early", "ended", "finished", "timed"), map(int, r.stdout.split())))

    return run


@pytest.mark.parametrize("seed", [1, 2])
def test_every_stage_is_consumed_without_a_timeout(model, seed):
    got = model(seed, -1, 1 << 20, 1 << 20)
    assert got == {"rearm": 0, "overlap": 0, "early": 0, "ended": 0, "finished": RUNS, "timed": 0}


@pytest.mark.parametrize("skip", [0, 1, 3])
# limits in polls: a copy lands within 60 steps of the model, so 300 polls of one agent outlast every copy
@pytest.mark.parametrize("lp,lc", [(300, 300), (300, 600), (600, 300)])
def test_a_stage_never_issued_leaves_no_copy_and_no_second_arrival(model, skip, lp, lc):
    got = model(11, skip, lp, lc)
    assert got["timed"] == RUNS and got["finished"] == 0
    assert (got["rearm"], got["overlap"], got["early"], got["ended"]) == (0, 0, 0, 0)


def test_waits_that_run_out_while_the_copies_are_on_their_way(model):
    got = model(21, -1, 300, 4)  # consumers give up on copies that do land
    assert got["timed"] > 0
    assert (got["rearm"], got["overlap"], got["early"], got["ended"]) == (0, 0, 0, 0)


def test_the_model_sees_buffers_handed_back_after_a_timeout(model):
    got = model(11, 1, 600, 300, plant=True)
    assert got["rearm"] > 0 and got["early"] > 0
