"""Contexts and runs without the device buffers that only make them faster (as when device memory is short):
the same chains and records, by the former kernels."""

import numpy as np
import pytest

import paper_1803_07030_gb300 as vg
from paper_1803_07030_gb300 import vegas as vb
from lattices import core_shell_particle, nanoparticle_batch, sc_periodic

pytestmark = pytest.mark.gpu

CASES = {
    "batch": (lambda: nanoparticle_batch(7, seed=4, r_max=7.0), 2, {}),
    "batch_blocks": (lambda: nanoparticle_batch(7, seed=4, r_max=7.0), 1, dict(variant=1, resident_smem=1)),
    "batch_clusters": (lambda: nanoparticle_batch(7, seed=4, r_max=7.0), 1,
                       dict(variant=3, resident_smem=1, cluster_blocks=2, cluster_threads=512)),
    "cooperative": (lambda: [core_shell_particle(3, radius=6.0, core_radius=4.0)], 4, dict(variant=2)),
    "fp64": (lambda: [sc_periodic(6)], 2, dict(variant=2, precision=64)),
    "automatic": (lambda: [sc_periodic(8)], 1, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_same_chain_without_spare_buffers(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    make, R, kw = CASES[name]
    samples = make()
    n = len(samples) * R
    T = np.linspace(0.5, 1.5, n)[:, None]
    with vg.Context(samples, replicas=R, seed=6, stream=None, **kw) as a, \
            vg.Context(samples, replicas=R, seed=6, stream=None, fault_inject=2, **kw) as b:
        for c in (a, b):
            c.run(T, 0.1, 40)
            c.run(T, 0.2, 9)
        assert b.stats()["tile_form"] == 0 and b.stats()["device_bytes"] < a.stats()["device_bytes"]
        for i in range(n):
            assert np.array_equal(a.spins(i), b.spins(i))
        assert np.array_equal(a.accept_history(), b.accept_history())
        bound = 64 * 2.0 ** -24 * 8.0 * max(s.n_sites for s in samples)  # FP32 runs of at most 64 attempts
        assert np.abs(a.history() - b.history()).max() <= bound


def test_other_values_are_refused():
    if not pytest.importorskip("torch").cuda.is_available():
        pytest.skip("no CUDA device")
    with pytest.raises(vb.VegasError) as e:
        vg.Context([sc_periodic(4)], fault_inject=3)
    assert e.value.status == vb.EINVAL


@pytest.mark.parametrize("variant, precision", [(0, 32), (0, 64), (1, 32), (3, 32)])
def test_a_fixed_sweep_keeps_no_other_sweep_s_tables(variant, precision):
    if not pytest.importorskip("torch").cuda.is_available():
        pytest.skip("no CUDA device")
    for samples in ([sc_periodic(8)], nanoparticle_batch(3, seed=2, r_max=5.0)):
        with vg.Context(samples, precision=precision, variant=variant, stream=None) as a, \
                vg.Context(samples, precision=precision, variant=variant, stream=None, fault_inject=2) as b:
            assert a.stats()["device_bytes"] == b.stats()["device_bytes"]
