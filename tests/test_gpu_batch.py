"""The batch kernel (spins in shared memory) over its dispatch: rows as words or pairs, parameter kinds,
whole blocks, groups of threads, clusters, instances without links and with several replicas. Spins,
accept log and counts equal the per-class sweep's bit for bit."""

import numpy as np
import pytest

import paper_1803_07030_gb300 as vg
from lattices import chain_open, core_shell_particle, fcc_sphere, free_spins, nanoparticle_batch, random_graph, sc_periodic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    vg.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _mixed():
    """Uneven instances: 1 to 4k sites, no links to full rows, uniaxial terms on some."""
    return [free_spins(1), chain_open(2), free_spins(300, k_uni=0.2, e_uni=(0, 1, 1)), sc_periodic(5), sc_periodic(12, k_uni=0.1),
            core_shell_particle(2, radius=6.0, core_radius=4.0), fcc_sphere(5.0), chain_open(513)]


def _graphs():
    return [random_graph(200, 0.02, s) for s in (3, 4)] + [fcc_sphere(3.0)]  # cubic terms, many exchange values


SETS = {"plain": (lambda: nanoparticle_batch(9, seed=3, r_max=9.0), 1), "mixed": (_mixed, 2), "graphs": (_graphs, 4)}
SHAPES = {
    "blocks": dict(variant=1, resident_smem=1),
    "groups_128": dict(variant=1, resident_smem=1, group_threads=128, group_sites=2048),
    "groups_256": dict(variant=1, resident_smem=1, group_threads=256, group_sites=100),
    "groups_64": dict(variant=1, resident_smem=1, group_threads=64, group_sites=500),
    "clusters_2": dict(variant=3, resident_smem=1, cluster_blocks=2, cluster_threads=512),
    "clusters_4_split": dict(variant=3, resident_smem=1, cluster_blocks=4, cluster_threads=512, cluster_split=400,
                             group_threads=256, group_sites=200),
    "automatic": dict(variant=-1),
}


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("name", list(SETS))
def test_batch_sweep_equals_per_class_sweep(name, shape):
    make, R = SETS[name]
    samples = make()
    n = len(samples) * R
    T = np.linspace(0.4, 2.0, n)[:, None] * np.array([1.0, 0.7])
    B = np.tile([[0.3, -0.1]], (n, 1))
    mcs = 30 if shape == "automatic" else 7
    with vg.Context(samples, replicas=R, seed=13, variant=0, accept_log_mcs=3, stream=None) as a, \
            vg.Context(samples, replicas=R, seed=13, accept_log_mcs=3, stream=None, **SHAPES[shape]) as b:
        for c in (a, b):
            c.run(T, B, mcs)
            c.run(T[:, 1:], B[:, 1:], 5)
        for i in range(n):
            assert np.array_equal(a.spins(i), b.spins(i)), i
        assert np.array_equal(a.accept_history(), b.accept_history())
        assert np.array_equal(a.accept_log(), b.accept_log())
        # FP32 runs of at most 64 attempts, then FP64, on both sides
        per_site = max(s.n_sites for s in samples)
        scale = max(1.0, np.abs(a.history()).max() / per_site)
        assert np.abs(a.history() - b.history()).max() <= 64 * 2.0 ** -24 * scale * per_site


def test_batches_of_different_sizes_in_turn():
    """Two batches whose blocks take different amounts of shared memory, run in turn."""
    p, q = nanoparticle_batch(3, seed=1, r_max=5.0), [fcc_sphere(14.0, a=4.0 ** (1.0 / 3.0))] * 2
    kw = dict(variant=1, resident_smem=1, seed=2, stream=None)
    with vg.Context(p, **kw) as a, vg.Context(q, **kw) as b, vg.Context(q, seed=2, variant=0, stream=None) as c:
        for k in range(2):
            b.run(1.0, 0.0, 4)
            a.run(1.0, 0.0, 4)
            c.run(1.0, 0.0, 4)
        assert np.array_equal(b.spins(1), c.spins(1))


def test_many_classes_keep_the_former_sums():
    """62 colour classes, 91 attempts per thread and MCS: the former kernels end a run of FP32 sums at 64."""
    s = sc_periodic((20, 20, 40))
    parity = np.asarray(vg.vegas_greedy_colour(s.row_ptr, s.col)[0])
    s.colour = np.where(np.arange(s.n_sites) < 60, 2 + np.arange(s.n_sites), parity).astype(np.int32)
    got = []
    for fault in (0, 2):  # 2: without the batch kernel's tables
        with vg.Context([s], seed=3, variant=1, resident_smem=1, fault_inject=fault, stream=None) as c:
            c.run(1.0, 0.1, 6)
            got.append((c.history(), c.spins(0)))
    assert np.array_equal(got[0][1], got[1][1])
    assert np.abs(got[0][0] - got[1][0]).max() <= 2.0 ** -50 * 8.0 * s.n_sites  # FP64 sums in another order
