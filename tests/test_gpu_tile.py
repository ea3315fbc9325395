"""The tiled cooperative sweep over its dispatch: part counts, rows kept as pairs or words, what fits
in shared memory, one and two FP32 buffers, parameters and policies. Spins, accept log and accepted
counts equal the per-class sweep's bit for bit (same attempts on the same random numbers), the
history to the FP32 partial sums' rounding."""

import numpy as np
import pytest

import paper_1803_07030_gb300 as vg
from lattices import chain_open, core_shell_particle, dimers, fcc_sphere, free_spins, random_graph, sc_periodic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    vg.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _sparse(seed):
    """Random rows of 0 to 12 links with every kind of term (over 32 exchange values)."""
    s = random_graph(300, 0.015, seed)
    assert np.diff(s.row_ptr).max() <= 12 and np.diff(s.row_ptr).min() == 0
    return s


CASES = {
    "one_site": (lambda: free_spins(1, field_axis=(0, 0, 1)), 1, {}),
    "no_links": (lambda: free_spins(777, k_uni=0.3, e_uni=(1, 0, 1)), 4, {}),
    "pairs_of_two": (lambda: dimers(100), 2, {}),
    "chain": (lambda: chain_open(1001), 1, {}),
    "odd_sides": (lambda: sc_periodic((5, 7, 9)), 1, {}),                   # three classes or more
    "one_block_per_replica": (lambda: sc_periodic(12), 32, {"max_blocks": 32}),
    "few_blocks": (lambda: sc_periodic(16, bimodal_seed=4), 2, {"max_blocks": 7}),
    "uniaxial": (lambda: sc_periodic(20, k_uni=0.2, e_axis=(1, 1, 0)), 1, {}),
    "core_shell": (lambda: core_shell_particle(5, radius=6.3, core_radius=4.0), 8, {}),
    "cubic_and_all_terms": (lambda: _sparse(3), 4, {}),
    "policies": (lambda: core_shell_particle(6, radius=5.0, core_radius=3.0).with_policy([4, 3], [0.5, 0.4]), 2, {}),
    "words_in_shared_memory": (lambda: sc_periodic((40, 40, 38), bimodal_seed=2), 8, {}),
    "words_through_l1": (lambda: sc_periodic((60, 60, 60), bimodal_seed=2), 8, {}),
    "pairs_through_l1": (lambda: fcc_sphere(20.0, a=4.0 ** (1.0 / 3.0)).with_policy([3], [0.4]), 16, {}),
    "one_buffer": (lambda: sc_periodic((128, 128, 126), bimodal_seed=2), 1, {}),
    "one_buffer_small_sample": (lambda: sc_periodic(30, bimodal_seed=2), 1, {"max_blocks": 2}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_tiled_sweep_equals_per_class_sweep(name):
    make, R, kw = CASES[name]
    s = make()
    big = s.n_sites * R > 500_000
    T = np.stack([np.array([1.6, 0.7]) * (1 + 0.1 * i) for i in range(R)])
    B = np.stack([np.array([0.5, -0.5]) for _ in range(R)])
    mcs = 3 if big else 8
    log = 0 if big else 3
    with vg.Context([s], replicas=R, seed=31, variant=0, accept_log_mcs=log, stream=None) as a, \
            vg.Context([s], replicas=R, seed=31, variant=2, accept_log_mcs=log, stream=None, **kw) as b:
        for c in (a, b):
            c.run(T[:, :1], B[:, :1], mcs)
            c.run(T[:, 1:], B[:, 1:], mcs)
        assert b.stats()["variant"] == 2
        for i in {0, R // 2, R - 1}:
            assert np.array_equal(a.spins(i), b.spins(i)), i
        assert np.array_equal(a.accept_history(), b.accept_history())
        if log:
            assert np.array_equal(a.accept_log(), b.accept_log())
        # both sides add FP32 runs of at most 64 attempts, then FP64: each term rounds to 2^-24 of a
        # run's partial sum, so 64 * 2^-24 of the largest site share bounds the difference per site
        scale = max(1.0, np.abs(a.history()[:, :, 0]).max() / s.n_sites)
        assert np.abs(a.history() - b.history()).max() <= 64 * 2.0 ** -24 * scale * s.n_sites


def test_long_step_in_several_launches():
    """More MCS per step than one launch takes (1024), and the counter set back in between: no
    mailbox word of an earlier pass over the same MCS is read."""
    s = sc_periodic(8)
    with vg.Context([s], replicas=2, seed=7, variant=0, stream=None) as a, \
            vg.Context([s], replicas=2, seed=7, variant=2, stream=None) as b:
        T = np.array([[0.9], [1.3]])
        for c in (a, b):
            c.run(T, 0 * T, 2100)
            c.set_mcs_counter(3)
            c.run(T, 0 * T, 40)
        for i in range(2):
            assert np.array_equal(a.spins(i), b.spins(i))
        assert np.array_equal(a.accept_history(), b.accept_history())


def test_contexts_of_different_sizes_in_turn():
    """Two contexts whose blocks take different amounts of shared memory run in turn."""
    p, q = fcc_sphere(9.0), sc_periodic(50)
    with vg.Context([p], seed=1, variant=2, stream=None) as a, vg.Context([q], seed=1, variant=2, stream=None) as b, \
            vg.Context([p], seed=1, variant=0, stream=None) as c:
        for k in range(3):
            a.run([[1.0]], [[0.1]], 5)
            b.run([[1.0]], [[0.1]], 5)
            c.run([[1.0]], [[0.1]], 5)
        assert np.array_equal(a.spins(0), c.spins(0))


@pytest.mark.parametrize("make, R", [(lambda: sc_periodic(8), 1), (lambda: sc_periodic(10), 32),
                                     (lambda: core_shell_particle(3, radius=8.0, core_radius=6.0), 1)])
def test_automatic_choice_keeps_the_chain(make, R):
    """The autotuner's first run (several sweeps in turn) and the runs after it."""
    s = make()
    T = np.linspace(0.5, 1.5, R)[:, None]
    with vg.Context([s], replicas=R, seed=5, stream=None) as a, vg.Context([s], replicas=R, seed=5, variant=0, stream=None) as b:
        for c in (a, b):
            c.run(T, 0 * T + 0.1, 60)
            c.run(T, 0 * T + 0.1, 7)
        for i in {0, R - 1}:
            assert np.array_equal(a.spins(i), b.spins(i))
        assert np.array_equal(a.accept_history(), b.accept_history())


FP64 = {
    "one_site": (lambda: free_spins(1, field_axis=(0, 0, 1)), 1, {}),
    "sc6_anisotropic": (lambda: sc_periodic(6, k_uni=0.3, e_axis=(1, 1, 0)), 2, {}),
    "odd_sides": (lambda: sc_periodic((5, 7, 9), bimodal_seed=1), 1, {}),
    "all_terms": (lambda: _sparse(8), 4, {}),
    "several_rounds": (lambda: sc_periodic(8, bimodal_seed=3), 32, {}),       # 64 sites of a class per part
    "two_blocks": (lambda: sc_periodic((4, 4, 6)), 1, {"max_blocks": 2}),
    "fcc": (lambda: fcc_sphere(4.2), 3 + 1, {}),
    "core_shell": (lambda: core_shell_particle(4, radius=5.0, core_radius=3.5), 1, {}),
}


@pytest.mark.parametrize("name", list(FP64))
def test_fp64_tiled_sweep_equals_oracle(name):
    import oracle

    make, R, kw = FP64[name]
    s = make()
    mcs = 6
    T = np.stack([[2.0 - 0.02 * r, 0.02, 0.6] for r in range(R)])  # a cold step: decisions far out in the tail
    B = np.stack([[0.3, -0.2, 0.1 * r] for r in range(R)])
    with vg.Context([s], precision=64, replicas=R, seed=9, variant=2, accept_log_mcs=3 * mcs, stream=None, **kw) as c:
        c.run(T, B, mcs)
        assert c.stats()["block_threads"] % 32 == 0 and c.stats()["block_threads"] > 32  # the tiled form
        ref = oracle.run(s, T, B, mcs, seed=9, log_mcs=3 * mcs, n_threads=R)
        assert ref["err"] == 0
        alog = c.accept_log().reshape(3 * mcs, R, -1)
        for r in range(R):
            assert np.array_equal(c.spins(r), ref["spins"][r]), r
            assert np.array_equal(alog[:, r], ref["accept_log"][r]), r
            assert np.array_equal(c.accept_history()[r], ref["accepted"][r]), r
            assert np.allclose(c.history()[r], ref["history"][r], rtol=1e-12, atol=1e-12 * s.n_sites * 8)


def test_fp64_long_step_and_counter_set_back():
    s = sc_periodic(6)
    T = np.array([[0.9], [1.3]])
    with vg.Context([s], precision=64, replicas=2, seed=7, variant=0, stream=None) as a, \
            vg.Context([s], precision=64, replicas=2, seed=7, stream=None) as b:
        for c in (a, b):
            c.run(T, 0 * T, 1100)
            c.set_mcs_counter(3)
            c.run(T, 0 * T, 40)
        for i in range(2):
            assert np.array_equal(a.spins(i), b.spins(i))
        assert np.array_equal(a.accept_history(), b.accept_history())
        assert np.allclose(a.history(), b.history(), rtol=1e-12, atol=1e-10)
