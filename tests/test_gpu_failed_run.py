"""A run that fails on host memory after the sweep leaves the records as they were, and reading them stays
inside the caller's buffer."""

import os
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes as C, resource
import numpy as np
import paper_1803_07030_gb300 as vg
from paper_1803_07030_gb300 import vegas as vb
from lattices import sc_periodic

R, mcs, steps = 4, 3, 40
T = np.full((R, steps), 1.0)
c = vg.Context([sc_periodic(48)], replicas=R, seed=3, variant=0, snapshots=True, graphs=False, stream=None)
c.run(T, 0 * T, mcs)
kept = c.history(), c.accept_history()
lib = vb.load_library()
vm = int(next(x for x in open("/proc/self/status") if x.startswith("VmSize")).split()[1]) * 1024
# the snapshots of 40 steps are 283 MB on the way to the host; a third of that is left
resource.setrlimit(resource.RLIMIT_AS, (vm + (96 << 20), resource.RLIM_INFINITY))
try:
    c.run(T, 0 * T, mcs)
    print("ran")
except vb.VegasError as e:
    print("failed", e.status)
resource.setrlimit(resource.RLIMIT_AS, (resource.RLIM_INFINITY, resource.RLIM_INFINITY))
n = C.c_size_t()
for fn, shape, dtype, old in ((lib.vegas_history, (R, -1, 4), np.float64, kept[0]),
                              (lib.vegas_accept_history, (R, -1), np.uint32, kept[1])):
    assert fn(c.ptr, None, 0, C.byref(n)) == 0 and n.value == old.size, (n.value, old.size)
    room = np.full(n.value + 8 * R * mcs * steps, 77, dtype=dtype)  # as much again as the failed run had
    assert fn(c.ptr, room.ctypes.data_as(C.c_void_p), n.value, C.byref(n)) == 0
    assert np.all(room[n.value:] == 77), "written past the buffer"
    assert np.array_equal(room[:n.value].reshape(shape), old)
c.run(T[:, :1], 0 * T[:, :1], mcs)  # and records go on behind them
assert np.array_equal(c.history()[:, :steps * mcs], kept[0]) and c.history().shape[1] == (steps + 1) * mcs
assert np.array_equal(c.snapshot(R - 1, steps), c.spins(R - 1))
print("records kept")
"""


def test_failed_run_leaves_the_records():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, PYTHONPATH=ROOT), capture_output=True,
                       text=True, timeout=120)
    assert p.returncode == 0, p.stdout + p.stderr
    assert "failed 2" in p.stdout and "records kept" in p.stdout, p.stdout
