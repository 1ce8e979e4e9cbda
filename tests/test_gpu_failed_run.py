"""A run that fails on its way (here: its stream is being captured, so the
wait at its end returns an error and none of its work is done) leaves the
state where it was, and the calls that read the state or go on from it take
the step from the device.  The odd number of steps would leave the readers on
the other of the two position buffers.

In a child process: a capture that was broken off leaves an error pending.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")
pytest.importorskip("paper_2002_07109_gb300.bounce")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import numpy as np, torch
from paper_2002_07109_gb300 import bounce
from paper_2002_07109_gb300.water import water_droplet_molecules

s = water_droplet_molecules(40, seed=3)
def context():
    c = bounce.from_system(s, seed=2, jump_coulomb=False)
    c.set_state(s.q, s.v)
    c.run(4, bounce.BOUNCE)
    return c
a, b = context(), context()
want = b.energies()
grad = b.gradient(bounce.GRAD_FULL)
hist = b.pair_histogram(0, 1, 8.0, 40)
side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
with torch.cuda.stream(side):
    graph.capture_begin(capture_error_mode="thread_local")
    try:
        a.run(3, bounce.BOUNCE, stream=side.cuda_stream)
        raise SystemExit("the run of a captured stream did not fail")
    except bounce.BounceError as e:
        assert "CUDA" in str(e), e
    try:
        graph.capture_end()
    except RuntimeError:
        pass
got = a.energies()
assert got["step"] == 4, got["step"]
for k in ("coulomb", "lj", "bond", "angle", "kinetic"):
    assert got[k] == want[k], (k, got[k], want[k])
assert np.array_equal(a.gradient(bounce.GRAD_FULL), grad)
assert np.array_equal(a.pair_histogram(0, 1, 8.0, 40), hist)
assert np.array_equal(a.get_state()[0], b.get_state()[0])
print("ok", flush=True)
"""


def test_readers_after_a_run_that_failed():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
