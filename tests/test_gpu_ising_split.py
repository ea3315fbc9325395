"""The Ising pass over its dispatch: threads per word position (by lattice and replicas) and
thresholds per replica (by the field), spins and history equal to the oracle's exactly.

With 152 SMs a word position is taken by one thread from 77,824 word positions of four replicas
on (each position: 32 sites of one colour), by two from half of that, by four, then eight."""

import numpy as np
import pytest

import oracle
import paper_1803_07030_gb300 as vg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    vg.build()
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("dims, L, R, J, h, T", [
    (2, 64, 4, 1.0, 0.0, 2.2),        # 8 threads per position, Z / 2 thresholds
    (2, 64, 12, -1.0, 0.7, 1.5),      # the same with a field: up to Z + 1
    (2, 128, 4, 1.0, 9.0, 0.02),      # every threshold 0 (never) or always
    (2, 448, 16, 0.5, 0.0, 1.0),      # 4
    (2, 576, 32, 1.0, -0.3, 2.5),     # 2
    (2, 1024, 20, 1.0, 0.0, 2.3),     # 1
    (3, 64, 4, 1.0, 0.0, 4.5),
    (3, 64, 8, -0.7, 1.4, 3.0),       # J sum = -h for some classes
    (3, 128, 12, 1.0, 0.1, 4.6),
])
def test_pass_matches_oracle(dims, L, R, J, h, T):
    Ts = np.stack([[T * (1.0 + 0.05 * r), T] for r in range(R)])
    hs = np.stack([[h * (r % 3), h] for r in range(R)])
    mcs = 2
    with vg.IsingContext(dims, L, J=J, replicas=R, seed=21 + L) as c:
        c.run(Ts, hs, mcs)
        ref = oracle.ising_run(dims, L, J, Ts, hs, mcs, seed=21 + L)
        assert np.array_equal(c.history(), ref["history"])
        for r in range(R):
            assert np.array_equal(c.spins(r), ref["spins"][r]), r
