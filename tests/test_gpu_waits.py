"""Waits that run out (a block that the host asks not to run): reported once per run, in every form of the
cooperative sweep."""

import time

import numpy as np
import pytest

import paper_1803_07030_gb300 as vg
from paper_1803_07030_gb300 import vegas as vb
from lattices import sc_periodic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    vg.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("precision", [32, 64])
def test_timeout_ends_the_run_s_later_launches(precision, graphs):
    """12 launches of 1024 MCS and three steps: the limit passes once, not once per launch."""
    s = sc_periodic(8)
    kw = dict(precision=precision, seed=1, variant=2, stream=None, graphs=graphs)
    with vg.Context([s], **kw) as c:
        c.run(np.array([[1.0]]), np.array([[0.0]]), 3)  # loads the kernels
    with vg.Context([s], timeout_ns=100_000_000, fault_inject=1, **kw) as c:
        t = time.perf_counter()
        with pytest.raises(vb.VegasError) as e:
            c.run(np.ones((1, 3)), np.zeros((1, 3)), 4096)
        took = time.perf_counter() - t
        assert e.value.status == vb.ETIMEOUT and c.stats()["device_error"] & 8
        assert 0.1 <= took < 0.5  # twelve limits are 1.2 s
