"""The allocation-free sweep in one launch (classes of at most 8192 attempts) against the same call on
many disjoint copies of the sample with the same Philox ids (one launch per class): spins bit for bit."""

import types

import numpy as np
import pytest

from conftest import noalloc_device_layout

import paper_1803_07030_gb300 as vg
from paper_1803_07030_gb300 import vegas as vb
from lattices import chain_open, fcc_sphere, random_graph, sc_periodic

pytestmark = pytest.mark.gpu

CASES = [  # sample, replicas, (k, kc)
    (lambda: chain_open(2), 32, (0.0, 0.0)), (lambda: chain_open(129), 1, (0.2, 0.0)), (lambda: sc_periodic(5), 2, (0.0, 0.0)),
    (lambda: fcc_sphere(4.0), 8, (0.3, -0.2)), (lambda: random_graph(60, 0.3, 2), 4, (0.0, 0.0)),  # rows beyond 12 links
    (lambda: sc_periodic(16), 2, (0.0, 0.0)), (lambda: sc_periodic(16), 4, (0.0, 0.1)),  # two rounds; four: 8192 attempts
]


@pytest.fixture(scope="module")
def torch():
    vg.build()
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    return t


def _copies(s, k):
    n, e = s.n_sites, int(s.row_ptr[-1])
    return types.SimpleNamespace(
        n_sites=n * k, J=np.tile(s.J, k), col=np.concatenate([s.col + n * i for i in range(k)]).astype(s.col.dtype),
        row_ptr=np.concatenate([[0]] + [s.row_ptr[1:] + e * i for i in range(k)]).astype(s.row_ptr.dtype))


def _sweeps(torch, s, ids, R, sp, start):
    lay = noalloc_device_layout(torch, s, start)
    out = torch.zeros((R, 4), dtype=torch.float64, device="cuda")
    site_id = (lay["site_id"] % ids).contiguous()
    T, B = np.linspace(0.4, 2.0, R), np.linspace(-0.3, 0.4, R)
    got = []
    for t in (0, 1, 2):
        vg.vegas_sweep_noalloc(lay["spins"].data_ptr(), lay["links"].data_ptr(), lay["row_ptr"].data_ptr(),
                               site_id.data_ptr(), s.n_sites, lay["colour_start"], R, 1.0 / T, B, site_params=sp, seed=6,
                               inst0=3, t=t, out_ptr=out.data_ptr())
        got.append(out.cpu().numpy().copy())
    spins = np.empty((s.n_sites, R, 4), dtype=np.float32)
    spins[lay["order"]] = lay["spins"].cpu().numpy()
    return spins, np.array(got), int(np.diff(lay["colour_start"]).max()) * R


@pytest.mark.parametrize("case", range(len(CASES)))
def test_one_launch_equals_a_launch_per_class(torch, case):
    make, R, (k, kc) = CASES[case]
    s = make()
    n = s.n_sites
    up = np.tile([0.6, 0.0, 0.8], (n, 1))
    sp = np.array([0.0, 0.6, 0.8, 1.0, 0.0, 0.0, 1.0, k, kc])
    one, sums, widest = _sweeps(torch, s, n, R, sp, [up] * R)
    assert widest <= 8192
    many = 8192 // widest + 1
    all_, sums_all, wide = _sweeps(torch, _copies(s, many), n, R, sp, [np.tile(up, (many, 1))] * R)
    assert wide > 8192
    assert np.array_equal(all_[:n], one) and np.array_equal(all_[-n:], one)
    # FP32 shares, added in FP64 on both sides
    assert np.abs(sums_all / many - sums).max() <= 1e-12 * max(1.0, np.abs(sums).max())


@pytest.mark.parametrize("side", [4, 30])  # one launch; a launch per class
def test_nan_is_reported(torch, side):
    s = sc_periodic(side)
    good = np.tile([0.0, 0.0, 1.0], (s.n_sites, 1))
    for bad in (False, True, False):
        if bad:
            with pytest.raises(vb.VegasError) as e:
                _sweeps(torch, s, s.n_sites, 1, None, [np.full_like(good, np.nan)])
            assert e.value.status == vb.EDEVICE
        else:
            _sweeps(torch, s, s.n_sites, 1, None, [good])
