"""Read passes at the edges of their kernels' tiles, against FP64 references.

  * the reduced density block on 1..3 qubits and the branch probabilities of
    channels on 1..6 qubits: states of exactly one gather set, of less than a
    staged tile (4096 amplitudes), of one tile and of several, below and above
    the sizes where the kernels change, with qubit 0 among the qubits or not,
    in unsorted order;
  * sampling where the cumulative table has more blocks than its scan has
    threads.

Tolerance of a density entry: FP32 products and runs of at most 32 sets (34
roundings of 2^-24), carried in double-floats, so |error| <= 36 * 2^-24 *
sqrt(rho_aa rho_bb); by Cauchy-Schwarz a probability is off by at most that
times |K|_F^2 N.  On 6 qubits, and below 2^18 sets, a wide channel's P_i are FP32 row sums of
2^q complex products, at most 4 * 64 roundings: 260 * 2^-24 of |K|_F^2 N.
"""
import numpy as np
import pytest

import qtsynth as qs
from gpu_util import random_state, to_device, torch_cuda

pytestmark = pytest.mark.gpu
EPS = 36 * 2.0 ** -24


@pytest.fixture(scope="module")
def qt():
    import paper_2111_02396_gb300 as pkg
    pkg.load()
    torch_cuda()
    return pkg


def density(psi, n, qubits):
    v = psi.astype(np.complex128).reshape([2] * n)       # axis i = qubit n - 1 - i
    front = [n - 1 - q for q in reversed(qubits)]
    rest = [i for i in range(n) if i not in front]
    m = v.transpose(front + rest).reshape(1 << len(qubits), -1)
    return m @ m.conj().T


CASES = [(1, 1), (2, 1), (2, 2), (3, 3), (4, 3), (12, 3), (13, 3), (17, 3), (9, 1), (13, 2), (4, 4), (5, 4), (12, 4),
         (15, 4), (5, 5), (6, 5), (13, 5), (16, 5), (6, 6), (7, 6), (12, 6), (13, 6), (17, 6),
         (22, 4), (23, 5), (24, 6), (23, 3), (23, 2)]


@pytest.mark.parametrize("n,q", CASES)
@pytest.mark.parametrize("low", [True, False])
def test_density_and_probabilities(qt, n, q, low):
    if not low and n == q:
        pytest.skip("every qubit is in the block")
    rng = np.random.default_rng([n, q, low])
    pool = np.arange(1, n)
    qubits = [int(x) for x in rng.choice(pool, q - 1 if low else q, replace=False)]
    if low:
        qubits.insert(int(rng.integers(q)), 0)
    psi = random_state(n, 50 + q) * np.float32(0.8)
    d = to_device(psi)
    ref = density(psi, n, qubits)
    N = np.trace(ref).real
    if q <= 3:
        rho = qt.qt_state_reduced_density(d.data_ptr(), n, qubits)
        p = np.sqrt(np.diag(ref).real)
        assert np.all(np.abs(rho - ref) <= EPS * np.outer(p, p) + 1e-300)
        np.testing.assert_array_equal(rho, rho.conj().T)
    Ks = qs.circuits.random_kraus(1 << q, 3, rng)
    P, got = qt.qt_state_kraus_probabilities(d.data_ptr(), n, qubits, Ks)
    assert abs(got - N) <= EPS * N
    for i, K in enumerate(Ks):
        want = np.trace(K.conj().T @ K @ ref).real
        tol = EPS if q <= 3 or (q <= 5 and n - q >= 18) else 260 * 2.0 ** -24
        assert abs(P[i] - want) <= tol * N * np.linalg.norm(K) ** 2, (i, P[i], want)


def test_sample_many_blocks(qt, orc):
    """2^27 amplitudes: 2048 blocks of the cumulative table, two per thread of its scan.
    Every sample lies in the neighbourhood of its target in C of the definition (FP64);
    the sampler's own C is off by at most 32 * 2^-24 of the total (FP32 squares and runs
    of at most 1024 terms)."""
    torch = torch_cuda()
    n, S = 27, 200
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    psi = torch.view_as_complex(torch.randn((1 << n, 2), generator=g, device="cuda"))
    got = qt.qt_state_sample(psi.data_ptr(), n, 9, 4, S).astype(np.int64)
    w = torch.view_as_real(psi).double()
    c = torch.cumsum((w * w).sum(1), 0)
    del w
    total = float(c[-1])
    t = np.array([orc.u01(9, 4, 1, j) for j in range(S)]) * total
    x = torch.tensor(got, device="cuda")
    above = c[x].cpu().numpy()
    below = torch.where(x > 0, c[(x - 1).clamp(min=0)], torch.zeros_like(c[x])).cpu().numpy()
    delta = 2 * 32 * 2.0 ** -24 * total
    assert np.all(t >= below - delta) and np.all(t <= above + delta)
