"""Thermal averages over the kernels' dispatch (chunks, bins and records behind them, lags per pass,
blocks per cluster) against the numpy oracle in FP64."""

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


@pytest.mark.parametrize("ns, length, cut, bins, tau", [
    (1, 2, 0, 2, 1.0),            # one record per bin, one lag
    (1, 40, 3, 7, 1.0),           # records behind the bins
    (3, 131, 100, 31, 2.0),
    (2, 1025, 1, 64, 3.0),        # two chunks of the load, most bins
    (1, 30000, 0, 20, 100.0),     # many lag passes, clusters of eight
    (20, 3000, 10, 33, 5.0),
    (77, 500, 100, 20, 4.0),      # no clusters
    (200, 333, 3, 10, 2.0),
])
def test_averages_match_oracle(ns, length, cut, bins, tau):
    rng = np.random.default_rng(ns + length)
    a = np.exp(-1.0 / tau)
    x = rng.normal(size=(length, ns, 4))
    for i in range(1, length):
        x[i] = a * x[i - 1] + np.sqrt(1 - a * a) * x[i]
    H = np.ascontiguousarray(np.swapaxes(x, 0, 1)) * np.array([20.0, 30.0, 30.0, 30.0]) + np.array([-3000.0, 0.0, 0.0, 200.0])
    T = np.linspace(0.5, 2.0, ns)
    out = vg.thermal_averages(H, cut, bins, T, 1000.0)
    for s in range(ns):
        ref = analysis.thermal_averages(H[s], cut, bins, T[s], 1000.0)
        for k, name in enumerate(vg.AVG_FIELDS):
            # sums of up to 30,000 centred terms in FP64, and differences of quantities 1e2 larger
            assert abs(out[s, k] - ref[name]) <= 1e-9 * abs(ref[name]) + 1e-9 * (3000.0 if name in ("v1", "v2") else 1e-3), (
                s, name, out[s, k], ref[name])


def test_constant_series_has_no_correlation_time():
    H = np.tile(np.array([-5.0, 0.0, 3.0, 4.0]), (2, 100, 1))
    out = vg.thermal_averages(H, 10, 5, 1.0, 10.0)
    assert np.allclose(out[:, [12, 13]], 0.5) and np.allclose(out[:, 0], -0.5) and np.allclose(out[:, 2], 0.5)


def test_constant_series_whose_sum_rounds():
    """n equal values whose sum is rounded have another plain mean: what is left after centring is zero."""
    rng = np.random.default_rng(7)
    for n, bins, values in ((8000, 20, (-1689.6, -921.6)), (800, 20, (-921.6, -0.1)), (1237, 10, tuple(-rng.uniform(1, 9e4, 60)))):
        H = np.empty((len(values), n, 4))
        H[:, :, 0] = np.array(values)[:, None]
        H[:, :, 1:] = (np.array(values) * 0.7)[:, None, None] * np.array([0.36, 0.48, 0.8])
        out = vg.thermal_averages(H, 0, bins, 1.3, 4096.0)
        assert np.array_equal(out[:, [12, 13]], np.full((len(values), 2), 0.5))


def test_squares_come_from_the_components():
    """M^2 of 2 and 12, whose roots round: 72 and 4 of 128 records (the others 0) give U4 = 0 exactly."""
    H = np.zeros((1, 128, 4))
    H[0, :, 0] = np.arange(128) % 3
    H[0, :72, 1:3] = 1.0
    H[0, 72:76, 1:] = 2.0
    out = vg.thermal_averages(H, 0, 4, 1.0, 10.0)
    assert out[0, vg.AVG_FIELDS.index("u4")] == 0.0
