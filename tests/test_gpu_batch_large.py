"""Batches beyond the sizes of the oracle tests, against the same trajectories in other batches.

Circuits without operations stay |0...0> and change nothing for the circuits around them.
"""
import numpy as np
import pytest

import qtsynth as qs
from gpu_util import torch_cuda
from test_gpu_batch import _noisy

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qt():
    import paper_2111_02396_gb300 as pkg
    pkg.load()
    torch_cuda()
    return pkg


@pytest.mark.parametrize("k", [3, 6])
def test_empty_circuits(qt, k):
    """The others' states, samples and records are those of a batch without the empty ones."""
    sizes = [3, 10, 11, 13, 14, 15]
    real = [qt.Fused(qt.Circuit.from_compact(_noisy(n, 5, n, 0.05)), k) for n in sizes]
    empty = {n: qt.Fused(qt.Circuit.from_synth(qs.Circuit(n)), k) for n in (1, 2, 12, 15)}
    alone = qt.Batch(real).run(seed=4, first_traj=100, samples_per_traj=20, keep_states=True)
    batch = [empty[1], real[0], empty[12], real[1], empty[15], real[2], empty[2], real[3], real[4], empty[15], real[5]]
    merged = qt.Batch(batch)
    for i, f in enumerate(batch):
        if f in real:                                        # with the trajectory id that it has alone
            j = real.index(f)
            b = merged.run(seed=4, first_traj=100 + j - i, samples_per_traj=20, keep_states=True)
            for x, y in zip(b.kraus_indices(i), alone.kraus_indices(j)):
                np.testing.assert_array_equal(x, y)
            np.testing.assert_array_equal(b.samples()[i], alone.samples()[j])
            np.testing.assert_array_equal(b.state(i), alone.state(j))
        else:
            b = merged.run(seed=4, samples_per_traj=20, keep_states=True)
            want = np.zeros_like(b.state(i))
            want[0] = 1.0
            np.testing.assert_array_equal(b.state(i), want)
            assert not np.any(b.samples()[i])
