"""Each form of the cooperative sweep, by what the context reports: the grid-barrier kernels (rows of six links,
padded rows, rows of any length, update policies) and the tiled ones by what a block keeps in shared memory.
Spins and counts equal the per-class sweep's bit for bit."""

import numpy as np
import pytest

import paper_1803_07030_gb300 as vg
from paper_1803_07030_gb300 import vegas as vb
from lattices import fcc_sphere, random_graph, sc_periodic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    vg.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _many_values(side):
    """A lattice with a thousand exchange values: its rows stay pairs."""
    s = sc_periodic(side)
    i = np.repeat(np.arange(s.n_sites), np.diff(s.row_ptr))
    s.J = 0.5 + ((i + s.col) * 7919 % 1009) / 1009.0
    return s


def _long_rows():
    s = random_graph(400, 0.06, 5)
    assert np.diff(s.row_ptr).max() > 12
    return s


def _fcc(r):
    return fcc_sphere(r, a=4.0 ** (1.0 / 3.0))


ROWS, IDS, NOTHING, WORDS, COLUMNS = 1 + 4, 1 + 2, 1, 8, 16
FORMS = {  # sample, replicas, tile_form (0: grid barriers)
    "barriers_six_links": (lambda: sc_periodic(22, bimodal_seed=1), 16, 0),
    "barriers_six_links_policy": (lambda: sc_periodic(22).with_policy([2], [0.4]), 16, 0),
    "barriers_padded_rows": (lambda: _fcc(14.0), 16, 0),
    "barriers_any_rows": (_long_rows, 4, 0),
    "one_round": (lambda: sc_periodic(20), 1, ROWS + COLUMNS),
    "one_round_padded_rows": (lambda: _fcc(14.0), 2, ROWS + COLUMNS),
    "pairs_in_shared_memory": (lambda: sc_periodic(64, k_uni=0.1), 1, ROWS),
    "words_in_shared_memory": (lambda: sc_periodic(80, bimodal_seed=2), 1, ROWS + WORDS),
    "words_through_l1": (lambda: sc_periodic(100, bimodal_seed=2), 1, IDS + WORDS),
    "padded_words_through_l1": (lambda: _fcc(45.0), 1, IDS + WORDS),
    "pairs_through_l1": (lambda: sc_periodic(100).with_policy([3], [0.4]), 1, IDS),
    "words_spins_alone": (lambda: sc_periodic(110), 1, NOTHING + WORDS),
    "pairs_spins_alone": (lambda: _many_values(110), 1, NOTHING),
}


@pytest.mark.parametrize("name", list(FORMS))
def test_form_equals_per_class_sweep(name):
    make, R, form = FORMS[name]
    s = make()
    T, B = np.linspace(0.7, 1.6, R)[:, None], np.full((R, 1), 0.3)
    with vg.Context([s], replicas=R, seed=8, variant=0, stream=None) as a, \
            vg.Context([s], replicas=R, seed=8, variant=2, stream=None) as b:
        for c in (a, b):
            c.run(T, B, 3)
            c.run(0.8 * T, -B, 3)
        assert b.stats()["tile_form"] == form and a.stats()["tile_form"] == 0
        for i in {0, R - 1}:
            assert np.array_equal(a.spins(i), b.spins(i)), i
        assert np.array_equal(a.accept_history(), b.accept_history())
        # FP32 runs of at most 64 attempts on both sides, as in the tiled sweep's own test
        scale = max(1.0, np.abs(a.history()[:, :, 0]).max() / s.n_sites)
        assert np.abs(a.history() - b.history()).max() <= 64 * 2.0 ** -24 * scale * s.n_sites


@pytest.mark.parametrize("make, R, precision, form", [
    (_long_rows, 32, 32, 0), (lambda: sc_periodic(22), 16, 32, 0), (lambda: _fcc(14.0), 16, 32, 0),
    (lambda: sc_periodic(12).with_policy([3], [0.4]), 1, 64, 0), (_long_rows, 1, 64, 0),
    (lambda: sc_periodic(12), 1, 32, ROWS + COLUMNS), (lambda: sc_periodic(12), 1, 64, 1)])
def test_a_block_that_does_not_come_is_reported(make, R, precision, form):
    with vg.Context([make()], replicas=R, precision=precision, seed=1, variant=2, timeout_ns=50_000_000, fault_inject=1,
                    stream=None) as c:
        with pytest.raises(vb.VegasError) as e:
            c.run(np.ones((R, 1)), np.zeros((R, 1)), 3)
        assert e.value.status == vb.ETIMEOUT and c.stats()["tile_form"] == form
        assert ("grid barrier" in str(e.value)) == (form == 0)


@pytest.mark.parametrize("make, R, kw, form", [(lambda: sc_periodic(8), 2, {}, 1), (lambda: sc_periodic(8), 32, {}, 1),
                                               (_long_rows, 1, {}, 0),
                                               (lambda: sc_periodic(6).with_policy([2], [0.5]), 1, {}, 0)])
def test_fp64_form(make, R, kw, form):
    with vg.Context([make()], replicas=R, precision=64, seed=1, variant=2, stream=None, **kw) as c:
        c.run(np.ones((R, 1)), np.zeros((R, 1)), 2)
        assert c.stats()["tile_form"] == form
