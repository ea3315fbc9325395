"""Rows of 32 replicas in planes (the per-class sweep's form): contexts where every sample, some or
none have it, changes of sweep, spins read and set in between, snapshots, policies. Spins equal
those of the sweep over whole instances, which keeps rows of float4, bit for bit."""

import numpy as np
import pytest

import paper_1803_07030_gb300 as vg
from lattices import chain_open, fcc_sphere, sc_periodic

pytestmark = pytest.mark.gpu


def _adaptive():
    s = sc_periodic(4)
    s.type = np.zeros(s.n_sites, dtype=np.int32)
    s.type_policy, s.type_param = np.array([vg.POLICY_ADAPTIVE], dtype=np.int32), np.array([0.5])
    return s


SETS = {
    "all": lambda: [sc_periodic(4), sc_periodic(6, k_uni=0.2)],
    "some": lambda: [chain_open(5), sc_periodic(4), fcc_sphere(2.0), sc_periodic(6, bimodal_seed=2)],
    "none": lambda: [fcc_sphere(2.5)],
    "one": lambda: [sc_periodic(8, bimodal_seed=1)],
    "adaptive": lambda: [_adaptive()],
}


@pytest.mark.parametrize("name", list(SETS))
def test_planar_rows(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    samples = SETS[name]()
    n = 32 * len(samples)
    T = np.linspace(0.4, 2.0, n)[:, None] * np.array([1.0, 0.8])
    kw = dict(replicas=32, seed=9, snapshots=1, stream=None)
    with vg.Context(samples, variant=0, **kw) as a, vg.Context(samples, variant=1, **kw) as b, \
            vg.Context(samples, **kw) as c:
        up = [np.tile([0.0, 0.6, 0.8], (s.n_sites, 1)) for s in samples]
        for mcs in (3, 40):  # the second is long enough for the automatic choice to be timed
            for x in (a, b, c):
                x.run(T, 0.1, mcs)
            for i in range(0, n, 7):
                want = b.spins(i)
                assert np.array_equal(a.spins(i), want) and np.array_equal(c.spins(i), want), (mcs, i)
            for x in (a, b, c):
                x.set_spins(n - 1, up[-1])
                assert np.array_equal(x.spins(n - 1), up[-1].astype(np.float32))
        for i in (0, n // 2, n - 1):
            for k in range(4):
                want = b.snapshot(i, k)
                assert np.array_equal(a.snapshot(i, k), want) and np.array_equal(c.snapshot(i, k), want), (i, k)
