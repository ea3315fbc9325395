"""The fused reweighting iteration over its dispatch (runs per call, samples per block) and the steps
it hands to the separate kernels, against the numpy oracle in FP64; and its exponential."""

import numpy as np
import pytest

from oracle import analysis
import paper_1803_07030_gb300 as vg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    vg.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _runs(K, n, sigma, gap, seed):
    """Gaussian density of states of width sigma, neighbouring betas gap / sigma apart."""
    rng = np.random.default_rng(seed)
    betas = 0.5 + np.arange(K) * gap / sigma
    E = rng.normal(size=(K, n)) * sigma - betas[:, None] * sigma ** 2
    return E, np.stack([E, (E / sigma) ** 2], axis=2), betas, np.linspace(betas[0], betas[-1], 5)


@pytest.mark.parametrize("K, n, sigma, gap", [
    (1, 100, 20.0, 1.0),
    (2, 1, 5.0, 0.5),            # one sample per run
    (3, 257, 20.0, 0.8),
    (4, 5000, 40.0, 0.9),
    (5, 1000, 40.0, 0.9),
    (8, 255, 30.0, 0.8),
    (9, 700, 30.0, 0.7),
    (16, 2049, 30.0, 0.6),
    (17, 300, 30.0, 0.6),        # more runs than the fused form takes
    (3, 2000, 400.0, 0.9),       # the first steps leave exp's range: taken by the separate kernels
])
def test_reweight_matches_oracle(K, n, sigma, gap):
    E, O, betas, targets = _runs(K, n, sigma, gap, 100 * K + n)
    out, g, it = vg.reweight(E, O, betas, targets, tol=1e-9)
    ref, gref, itref = analysis.reweight(E, O, betas, targets, tol=1e-9)
    # both stop within tol of the fixed point at the same step up to rounding: g is a logarithm of
    # sums relative to |beta E|'s rounding
    scale = np.abs(betas.max() * E).max() * 2.0 ** -52
    assert abs(it - itref) <= 1
    assert np.allclose(g, gref, rtol=0, atol=1e-8 + 64 * scale)
    assert np.allclose(out, ref, rtol=1e-8 + 64 * scale, atol=1e-9)


def test_max_iter_and_tight_tolerance():
    E, O, betas, targets = _runs(6, 900, 30.0, 0.9, 1)
    for m in (1, 15, 16, 17, 40):
        g, it = vg.reweight(E, O, betas, targets, max_iter=m, tol=1e-300)[1:]
        gref, itref = analysis.reweight(E, O, betas, targets, max_iter=m, tol=1e-300)[1:]
        assert it == itref == m
        assert np.allclose(g, gref, rtol=0, atol=1e-10)
