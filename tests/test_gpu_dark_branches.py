"""Branch probabilities of wide channels on states near the kernel of an operator, against FP64.

The state is a vector v on the channel's qubits times a uniform state on the others, so
that every gather set is the same and no rounding averages out.  K_0 = I - |u><u| with u
close to v: true P_0 from 0 to 1 (of N), by cancellation.  The other operators have no
small probability or none that cancels.

Tolerance: a row of K_i v is a sum of 2^q complex products of FP32 operands, off by at most
(2 2^q + 2) 2^-24 sum |k||v|, so |K_i v| is off by d = (2 2^q + 2) 2^-24 |K_i|_F |v|; the
squares and their runs of 16 sets add (2 2^q + 18) 2^-24 of P.  So |P - P_true| <= 2 sqrt(P_true) d +
d^2 + (2 2^q + 18) 2^-24 P_true.  Without cancellation (E_i <= P_i) a probability from the
density block is off by at most 13 roundings an entry, 14 * 2^-24 sum |G_ab||v_a||v_b| <=
14 * 2^-24 |K_i|_F^2 N, and of the order of a few 2^-24 P.
"""
import numpy as np
import pytest

from gpu_util import to_device, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qt():
    import paper_2111_02396_gb300 as pkg
    pkg.load()
    torch_cuda()
    return pkg


def _vector(d, rng):
    v = rng.standard_normal(d) + 1j * rng.standard_normal(d)
    return v / np.linalg.norm(v)


def _state(n, qubits, v):
    x = np.arange(1 << n, dtype=np.uint32)
    m = np.zeros(1 << n, np.uint8)
    for b, q in enumerate(qubits):
        m |= (((x >> q) & 1) << b).astype(np.uint8)
    return (v * 2.0 ** (-(n - len(qubits)) / 2)).astype(np.complex64)[m]


@pytest.mark.parametrize("n,qubits", [(22, (3, 0, 9, 8)), (23, (21, 5, 12, 7)), (24, (19, 20, 21, 22)),
                                      (23, (2, 3, 0, 22, 1)), (25, (4, 11, 19, 12, 7)), (24, (6, 0, 12, 18, 23, 1)),
                                      (16, (3, 9, 2, 15)), (17, (16, 1, 8, 4, 5))])
@pytest.mark.parametrize("true", [0.0, 1e-9, 1e-8, 1e-6, 1e-3, 0.3, 1.0])
def test_near_dark_branch(qt, n, qubits, true):
    q = len(qubits)
    D = 1 << q
    rng = np.random.default_rng([n, q, int(true * 1e9)])
    u, w = _vector(D, rng), _vector(D, rng)
    w -= np.vdot(u, w) * u
    w /= np.linalg.norm(w)
    # K_0 of complex64 operands; v in its kernel up to their rounding
    K0 = (np.eye(D) - np.outer(u, u.conj())).astype(np.complex64).astype(np.complex128)
    one = np.zeros((D, D), complex)
    one[1, int(rng.integers(D))] = 0.01
    mixed = 0.5 * np.linalg.qr(rng.standard_normal((D, D)) + 1j * rng.standard_normal((D, D)))[0]
    Ks = np.stack([K0, one.astype(np.complex64), mixed.astype(np.complex64)]).astype(np.complex128)
    v = np.sqrt(1 - true) * u + np.sqrt(true) * w
    psi = _state(n, qubits, 0.9 * v)
    # the FP32 vector itself, in 64 bits
    f = (0.9 * v * 2.0 ** (-(n - q) / 2)).astype(np.complex64).astype(np.complex128) * 2.0 ** ((n - q) / 2)
    N = np.vdot(f, f).real
    P, got = qt.qt_state_kraus_probabilities(to_device(psi).data_ptr(), n, list(qubits), Ks)
    eps = 2.0 ** -24
    assert abs(got - N) <= (2 * D + 18) * eps * N
    for i, K in enumerate(Ks):
        want = np.linalg.norm(K @ f) ** 2
        d = (2 * D + 2) * eps * np.linalg.norm(K) * np.sqrt(N)
        assert P[i] >= 0.0
        assert abs(P[i] - want) <= 2 * np.sqrt(want) * d + d * d + (2 * D + 18) * eps * want, (i, P[i], want)
