"""Sweeps that give a thread the same sites record the same sums, whatever kernel runs: equal spins, and
histories to the FP64 sums' rounding (n terms of 2^-53 each; the FP32 sums of another order are 1e4 times
further apart)."""

import numpy as np
import pytest

import paper_1803_07030_gb300 as vg
from lattices import sc_periodic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    vg.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _records(s, R, kw, T, runs=2):
    with vg.Context([s], replicas=R, seed=17, stream=None, **kw) as c:
        t = np.linspace(T, 1.5 * T, R)[:, None]
        for _ in range(runs):
            c.run(t, 0 * t + 0.1, 40)
        return c.spins(R - 1), c.history()[:, -40:], c.accept_history(), c.stats()


def _near(a, b, s):
    return np.abs(a - b).max() <= 2.0 ** -50 * 8.0 * s.n_sites


PAIRS = {  # sites of a class at once, on both sides
    "resident_512": (11, 1, dict(variant=1, resident_smem=1), dict(variant=2, max_blocks=2)),
    "resident_256": (11, 1, dict(variant=1, resident_smem=-1), dict(variant=2, max_blocks=1)),
    # a part of the cooperative sweep's tiled form would take several rounds: the grid-barrier form stays
    "cluster_1024": (16, 16, dict(variant=3, resident_smem=-1, cluster_blocks=4, cluster_threads=256),
                     dict(variant=2, max_blocks=64)),
    "cluster_1024_32": (16, 32, dict(variant=3, resident_smem=-1, cluster_blocks=4, cluster_threads=256),
                        dict(variant=2, max_blocks=128)),
    # a thread per site: the tiled form
    "whole_class": (12, 1, dict(variant=3, resident_smem=1, cluster_blocks=2, cluster_threads=512), dict(variant=2)),
    "batch_and_former_kernel": (14, 4, dict(variant=1, resident_smem=1),
                                dict(variant=1, resident_smem=-1, group_threads=0)),
}


@pytest.mark.parametrize("name", list(PAIRS))
def test_same_sites_per_thread_same_records(name):
    side, R, a, b = PAIRS[name]
    s = sc_periodic((side, side, side + 1 if R == 1 else side), bimodal_seed=5)
    if name == "batch_and_former_kernel":
        s = sc_periodic((16, 16, 17))  # 4352 sites: the resident sweep takes 512 threads in both forms
    x, y = _records(s, R, a, 0.8), _records(s, R, b, 0.8)
    assert np.array_equal(x[0], y[0]) and np.array_equal(x[2], y[2])
    assert _near(x[1], y[1], s)


@pytest.mark.parametrize("sides, R, policy", [((11, 14, 11), 1, 2), ((9, 10, 8), 1, None), ((22, 22, 22), 16, None),
                                              ((16, 20, 17), 1, None), ((12, 12, 12), 8, None)])
def test_automatic_records_are_those_of_a_timed_sweep(sides, R, policy):
    """The second run of an automatic context records what one of the sweeps does that its first run timed."""
    s = sc_periodic(sides, bimodal_seed=3)
    if policy is not None:
        s.with_policy(policy, 0.5)
    x = _records(s, R, {}, 0.9)
    per_sm = [dict(variant=2, max_blocks=152 * k) for k in (1, 2, 3)]
    resident = [dict(variant=1, resident_smem=1), dict(variant=1, resident_smem=-1), dict(variant=2, max_blocks=max(1, R)),
                dict(variant=2, max_blocks=2 * R)]
    clusters = [dict(variant=3, resident_smem=-1, cluster_blocks=cs, cluster_threads=256) for cs in (2, 4, 8, 16)]
    others = [_records(s, R, kw, 0.9) for kw in [dict(variant=0)] + per_sm + resident + clusters]
    for y in others:
        assert np.array_equal(x[0], y[0]) and np.array_equal(x[2], y[2])
    assert any(_near(x[1], y[1], s) for y in others), x[3]["variant"]
