"""Records reach the host by instance: several runs, one and many instances, large histories."""

import numpy as np
import pytest

import paper_1803_07030_gb300 as vg
from lattices import chain_open

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_inst, mcs", [(1, (5, 3)), (3, (1, 4, 2)), (257, (4, 700))])  # 257 x 704: several host threads
def test_records_by_instance_over_runs(n_inst, mcs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    samples = [chain_open(2 + i % 41) for i in range(n_inst)]
    T = np.linspace(0.5, 1.5, n_inst)[:, None]
    with vg.Context(samples, seed=4, stream=None) as c:
        done = 0
        for n in mcs:
            c.run(T, 0.2, n)
            before = c.history()[:, :done], c.accept_history()[:, :done]
            if done:
                assert np.array_equal(before[0], kept[0]) and np.array_equal(before[1], kept[1])
            done += n
            kept = c.history(), c.accept_history()
            assert kept[0].shape == (n_inst, done, 4) and kept[1].shape == (n_inst, done)
            for i, s in enumerate(samples):  # a chain of unit spins: M is their sum, FP32 rounding per MCS
                m = c.spins(i).reshape(-1, 3).sum(0, dtype=np.float64)
                assert np.abs(kept[0][i, -1, 1:] - m).max() <= 2.0 ** -22 * s.n_sites * done
                assert kept[1][i].max() <= s.n_sites
