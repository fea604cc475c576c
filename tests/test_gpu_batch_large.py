"""Batches that the oracle tests are too small for, against the same trajectories in other batches.

Circuits without operations stay |0...0> and change nothing for the circuits around them;
a trajectory's records and samples do not depend on the batch it runs in, nor on the CTAs
that its cluster has or the slot that it reuses.
"""
import numpy as np
import pytest

import qtsynth as qs
from gpu_util import MARGIN, torch_cuda
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


@pytest.mark.parametrize("k,per_sm", [(3, 2.1), (4, 2.1), (3, 1.3), (2, 0.6)])
def test_global_states_in_reused_slots(qt, orc, k, per_sm):
    """States in global memory, not kept, in batches of more than two, one to two, and less than one
    trajectory per SM (clusters of one, two and several CTAs), where a cluster takes trajectory after
    trajectory into its slot: the records and samples of the same trajectory ids in batches of eight."""
    torch = torch_cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    ccs = [_noisy(n, 4, s, 0.08) for s, n in enumerate([15, 16, 15, 17, 16, 15, 16])]
    fs = qt.fuse_many([qt.Circuit.from_compact(c) for c in ccs], k)
    num = int(sms * per_sm)
    S, first = 33, 700
    fused = [fs[i % len(fs)] for i in range(num)]
    big = qt.Batch(fused)
    big.run(seed=8, first_traj=first, samples_per_traj=S)
    assert big.stats()["flushes"] > num // 2
    for i0 in list(range(0, 24, 8)) + list(range(num // 2, num // 2 + 16, 8)) + [num - 16, num - 8]:
        small = qt.Batch(fused[i0:i0 + 8]).run(seed=8, first_traj=first + i0, samples_per_traj=S)
        np.testing.assert_array_equal(big.samples()[i0:i0 + 8], small.samples())
        for j in range(8):
            for x, y in zip(big.kraus_indices(i0 + j), small.kraus_indices(j)):
                np.testing.assert_array_equal(x, y)
    for i in (3, num // 2, num - 1):                         # and the oracle's, off ties
        ref = orc.run_trajectory(ccs[i % len(ccs)].to_circuit(), orc.DELAYED, seed=8, traj=first + i)
        kr, st = big.kraus_indices(i)
        tie = np.nonzero(ref["margin"] <= MARGIN)[0]
        upto = tie[0] if len(tie) else len(kr)
        np.testing.assert_array_equal(kr[:upto], ref["kraus_idx"][:upto])
        np.testing.assert_array_equal(st[:upto], ref["stage"][:upto])
        if not len(tie):
            want, margin = orc.sample(ref["state"], 8, first + i, S)
            ok = margin > MARGIN
            np.testing.assert_array_equal(big.samples()[i][ok], want[ok])
