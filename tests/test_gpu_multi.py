"""Passes of several fused gates: edges of the tile, against an FP64 product and against
one pass per gate.

A tile holds 12 qubits, so 12 -> 13 is where a state becomes several tiles (and the
launch changes from 512 to 128 threads); a pass takes 48 gates or the matrix entries that
its parameters hold, in a small (512) and a large form.

Tolerance: a gate of width k is a sum of 2^k complex products, each of three real ones
with sums of two entries as factors, so its error is at most 4 * 2^k * 2^-24 of the norm,
and an FP32 rounding of its matrix 2^k * 2^-24; over G fused gates 5 G 2^k 2^-24.
"""
import numpy as np
import pytest

import qtsynth as qs
from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qt():
    import paper_2111_02396_gb300 as pkg
    pkg.load()
    torch_cuda()
    return pkg


def _gates(n, widths, seed, near=False):
    """Random unitary gates of the given widths; near: on neighbouring qubits."""
    rng = np.random.default_rng([0x4D, n, seed])
    out = []
    for w in widths:
        q0 = int(rng.integers(0, n - w + 1))
        q = list(range(q0, q0 + w)) if near else sorted(int(x) for x in rng.choice(n, w, replace=False))
        u = np.linalg.qr(rng.normal(size=(1 << w, 1 << w)) + 1j * rng.normal(size=(1 << w, 1 << w)))[0]
        out.append((q, u))
    return out


def _circuit(n, gates):
    c = qs.Circuit(n)
    for i, (q, u) in enumerate(gates):
        c.gate(u, tuple(q), i)
    return c


def _exact(n, gates):
    psi = np.zeros(1 << n, np.complex128)
    psi[0] = 1.0
    for q, u in gates:
        w = len(q)
        t = psi.reshape((2,) * n)                            # axis n - 1 - i is qubit i
        ax = [n - 1 - x for x in reversed(q)]
        t = np.tensordot(u.reshape((2,) * (2 * w)), t, axes=(list(range(w, 2 * w)), ax))
        psi = np.ascontiguousarray(np.moveaxis(t, list(range(w)), ax)).ravel()
    return psi


@pytest.mark.parametrize("n", [8, 9, 10, 11, 12, 13, 14, 17, 20])
@pytest.mark.parametrize("k,count,near", [(1, 9, False), (2, 7, False), (2, 130, False), (3, 40, True), (4, 3, True),
                                          (4, 60, False)])
def test_against_fp64(qt, n, k, count, near):
    rng = np.random.default_rng([n, k, count])
    gates = _gates(n, [int(rng.integers(1, min(k, 2 if not near else k) + 1)) for _ in range(count)], k, near)
    run = qt.Run(qt.Fused(qt.Circuit.from_synth(_circuit(n, gates)), k), 1, keep_states=True)
    st = run.stats()
    ref = _exact(n, gates)
    got = run.state(0).astype(np.complex128)
    assert np.linalg.norm(got - ref) <= 5 * count * 2**k * 2.0**-24
    if n >= 8 + k and count > 30:
        assert st["fused_passes"] < st["fused_pieces"]


@pytest.mark.parametrize("n", [8, 9, 10, 11])
@pytest.mark.parametrize("k,count", [(1, 8), (2, 60), (3, 20), (3, 40), (4, 2), (4, 12)])
def test_same_sums_as_single_passes(qt, n, k, count):
    """One pass for each fused gate (full width, so none merge), in the plan's order, gives the same bits
    up to the run's normalization: an FP32 factor and a rounded product, 2^-24 each."""
    import torch
    gates, last = [], None
    for q, u in _gates(n, [k] * (2 * count), 77 + k):
        if q != last and len(gates) < count and (k > 1 or q[0] not in [g[0][0] for g in gates]):
            gates.append((q, u))
            last = q
    fused = qt.Fused(qt.Circuit.from_synth(_circuit(n, gates)), k)
    run = qt.Run(fused, 1, keep_states=True)
    num = fused.info()["num_fused"]
    assert run.stats()["fused_pieces"] == num >= len(gates) - 4
    psi = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
    psi[0] = 1.0
    for i in range(num):
        g = fused.gate(i)                                    # in the order of the plan
        qt.qt_state_apply(psi.data_ptr(), n, g["targets"], g["matrix"], stream=torch.cuda.current_stream().cuda_stream)
    a, b = run.state(0).view(np.float32).astype(np.float64), psi.cpu().numpy().view(np.float32).astype(np.float64)
    np.testing.assert_allclose(a, b / np.linalg.norm(b), rtol=2.0**-23 * 1.1, atol=0)
