"""Read passes on caller-owned states whose norm^2 leaves FP32's range while their amplitudes
and short sums of squares do not: |a|^2 around 3e34 (sums of a thousand stay below 2^128) and
around 1e-30, against FP64.

Tolerances are those of the same calls at norm 1: a density entry 36 * 2^-24 sqrt(rho_aa rho_bb),
a probability 260 * 2^-24 |K|_F^2 N, an expectation 2 * 135 * 2^-24 (FP32 runs of at most 128
amplitudes, their squares and sums).
"""
import numpy as np
import pytest

import qtsynth as qs
from gpu_util import random_state, to_device, torch_cuda
from test_gpu_reductions import EPS, density
from test_zz_no_alloc import _noalloc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qt():
    import paper_2111_02396_gb300 as pkg
    pkg.load()
    torch_cuda()
    return pkg


def _state(n, scale):
    return (random_state(n, 3) * np.float32(2.0 ** (n / 2))) * np.float32(scale)


@pytest.mark.parametrize("scale", [1.7e17, 1e-15])
@pytest.mark.parametrize("n,qubits", [(17, [4]), (17, [0, 16]), (17, [9, 3, 11]), (15, [0, 2, 7]), (15, [5, 1, 9, 2]),
                                      (16, [0, 3, 8, 12, 5]), (22, [2, 15, 3, 8]), (15, [1, 2, 4, 8, 10, 12]),
                                      (16, [0, 2, 4, 8, 10, 12])])
def test_density_and_probabilities(qt, n, qubits, scale):
    psi = _state(n, scale)
    d = to_device(psi)
    ref = density(psi, n, qubits)
    N = np.trace(ref).real
    assert scale < 1 or N > 2.0**128 * 1.5
    if len(qubits) <= 3:
        p = np.sqrt(np.diag(ref).real)
        for rho in (qt.qt_state_reduced_density(d.data_ptr(), n, qubits),
                    _noalloc(qt.load(), d.data_ptr(), n, qubits)):
            assert np.all(np.abs(rho - ref) <= EPS * np.outer(p, p))
    rng = np.random.default_rng(n)
    Ks = qs.circuits.random_kraus(1 << len(qubits), 3, rng)
    P, got = qt.qt_state_kraus_probabilities(d.data_ptr(), n, qubits, Ks)
    assert abs(got - N) <= 260 * 2.0**-24 * N
    for i, K in enumerate(Ks):
        want = np.trace(K.conj().T @ K @ ref).real
        assert abs(P[i] - want) <= 260 * 2.0**-24 * N * np.linalg.norm(K) ** 2


@pytest.mark.parametrize("scale", [1.7e17, 1e-15])
@pytest.mark.parametrize("n", [14, 16, 17, 20])
def test_expectations(qt, n, scale):
    psi = _state(n, scale)
    rng = np.random.default_rng(n)
    masks = [1 << q for q in range(n)] + [int(x) for x in rng.integers(1, 1 << n, 9)]
    z = qt.qt_state_expect_z(to_device(psi).data_ptr(), n, masks)
    w = np.abs(psi.astype(np.complex128)) ** 2
    x = np.arange(1 << n, dtype=np.uint64)
    for m, got in zip(masks, z):
        par = np.bitwise_count(x & np.uint64(m)) & 1
        want = (w[par == 0].sum() - w[par == 1].sum()) / w.sum()
        assert abs(got - want) <= 2 * 135 * 2.0**-24


def test_beyond_fp32(qt):
    """Amplitudes whose squares overflow by themselves are not finite, as before; a NaN stays one."""
    psi = _state(13, 1.0)
    psi[5] = 1e25
    rho = qt.qt_state_reduced_density(to_device(psi).data_ptr(), 13, [0, 3])
    assert not np.isfinite(rho[1, 1].real) and np.isfinite(rho[0, 0].real)
    psi[5] = np.nan
    assert np.isnan(qt.qt_state_expect_z(to_device(psi).data_ptr(), 13, [1])).all()
