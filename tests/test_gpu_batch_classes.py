"""Edges of the batched form's classes of shared-memory states, against the FP64 oracle.

The classes change at 10/11, 12/13, 13/14 and 14/15 qubits (CTA size and shared
memory); states of fewer than 32 amplitudes have sampling ranges past their end.
Also: more flush points than the list of them holds (64), more fused gates than a
descriptor window (128), pieces of more members than their list (64), and sample
counts around a warp's batch.  Tolerances are those of the other batch tests (state
2e-5, records and samples off ties).
"""
import numpy as np
import pytest

import qtsynth as qs
from gpu_util import torch_cuda
from test_gpu_batch import _noisy, check_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qt():
    import paper_2111_02396_gb300 as pkg
    pkg.load()
    torch_cuda()
    return pkg


def _chain(n, depth, seed, ad):
    rng = np.random.default_rng([0x81, n, depth, seed])
    return qs.layered_compact(n, depth, rng, lambda l: qs.circuits._chain_couplings(n, l), dep1=0.02, per_gate_ad=ad)


@pytest.mark.parametrize("k,threads,S", [(1, 512, 1), (3, 512, 33), (3, 128, 600), (4, 256, 8), (6, 128, 7)])
def test_class_edges(qt, orc, k, threads, S):
    ccs = [_noisy(n, 6, s, 0.05) for s, n in enumerate([2, 3, 4, 5, 6, 10, 11, 12, 13, 14, 15])]
    b, _ = check_batch(qt, orc, ccs, k, seed=21, first=10, S=S, threads=threads)
    assert b.stats()["flushes"] > 0


def test_one_qubit_states(qt, orc):
    c = qs.Circuit(1)
    for m in range(0, 12, 3):
        c.gate(qs.SQRT_X if m % 2 else qs.SQRT_W, (0,), m)
        c.channel(qs.amplitude_damping(0.2), (0,), m + 1)
        c.channel(qs.phase_damping(0.1), (0,), m + 2)
    f = qt.Fused(qt.Circuit.from_synth(c), 1)
    b = qt.Batch([f] * 6).run(seed=2, samples_per_traj=40, keep_states=True)
    r = qt.Run(f, 6, seed=2, samples_per_traj=40, keep_states=True)
    for i in range(6):
        np.testing.assert_array_equal(b.kraus_indices(i)[0], r.kraus_indices()[0][i])
        np.testing.assert_allclose(b.state(i), r.state(i), atol=2e-6)
        np.testing.assert_array_equal(b.samples()[i], r.samples()[i])


def test_many_flushes(qt, orc):
    """More than 64 undecided channels in a trajectory."""
    ccs = [_chain(n, 40, n, 0.5) for n in (5, 6, 7)]
    b, _ = check_batch(qt, orc, ccs, 2, seed=5, S=16)
    st = b.stats()
    assert st["flushes"] > 3 * 64


@pytest.mark.parametrize("k", [2, 5])
def test_deep_circuits(qt, orc, k):
    """More than 128 fused gates (k = 2), pieces of more than 64 members (k = 5)."""
    ccs = [_chain(n, 90, n, 2e-3) for n in (7, 9)]
    _, fs = check_batch(qt, orc, ccs, k, seed=6, S=16)
    if k == 2:
        assert max(f.info()["num_fused"] for f in fs) > 128
    else:
        assert max(len(f.gate(g)["members"]) for f in fs for g in range(f.info()["num_fused"])) > 64
