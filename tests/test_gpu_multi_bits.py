"""k_multi against one pass per gate, the same bits: raw floats of a random un-normalized
state, for gates of width 1 to 4, one tile and many tiles, and every size of the kernel's
parameters (up to 512, 1024 and 2176 matrix entries), through the launchers themselves.
"""
import ctypes as C

import numpy as np
import pytest

from gpu_util import random_state, to_device, torch_cuda

pytestmark = pytest.mark.gpu


class MultiPiece(C.Structure):
    _fields_ = [("k", C.c_int), ("targets", C.c_uint32 * 4), ("u", C.c_void_p)]


@pytest.fixture(scope="module")
def lib():
    import paper_2111_02396_gb300 as pkg
    torch_cuda()
    lib = pkg.load()
    lib.multi = getattr(lib, "_ZN2qt12launch_multiEP6float2iiPKNS_10MultiPieceEP11CUstream_st")
    lib.multi.argtypes = [C.c_void_p, C.c_int, C.c_int, C.POINTER(MultiPiece), C.c_void_p]
    lib.apply = getattr(lib, "_ZN2qt12launch_applyEP6float2iiPKjPKS0_P11CUstream_st")
    lib.apply.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]
    return lib


CASES = [(n, widths, low) for n in (8, 9, 10, 11, 12, 13, 14, 17, 21)
         for widths in ([1] * 48, [2] * 32, [2] * 48, [3] * 8, [3] * 16, [3] * 33, [4] * 2, [4] * 4, [4] * 8,
                        [1, 4, 2, 3, 3, 1, 2, 4, 1], [1])
         for low in (False, True) if n >= 7 + max(widths)]


@pytest.mark.parametrize("n,widths,low", CASES, ids=[f"n{n}-{len(w)}x{max(w)}{'-low' if x else ''}" for n, w, x in CASES])
def test_same_bits(lib, n, widths, low):
    """low: qubits of the tile are the lowest; otherwise they lie anywhere."""
    torch = torch_cuda()
    rng = np.random.default_rng([n, len(widths), max(widths), low])
    pool = np.arange(n) if n <= 12 else (np.arange(12) if low else np.concatenate(
        [np.arange(4), rng.choice(np.arange(4, n), 8, replace=False)]))
    pieces, mats = (MultiPiece * len(widths))(), []
    for i, w in enumerate(widths):
        q = sorted(int(x) for x in rng.choice(pool, w, replace=False))
        u = (rng.standard_normal((1 << w, 1 << w)) + 1j * rng.standard_normal((1 << w, 1 << w))) * 2.0 ** (-w / 2)
        mats.append(np.ascontiguousarray(u.astype(np.complex64)))
        pieces[i] = MultiPiece(w, (C.c_uint32 * 4)(*q), mats[-1].ctypes.data)
    start = to_device(random_state(n, 8) * np.float32(1.3))
    one, many = start.clone(), start.clone()
    assert lib.multi(many.data_ptr(), n, len(widths), pieces, None) == 0
    for p in pieces:
        assert lib.apply(one.data_ptr(), n, p.k, C.byref(p, MultiPiece.targets.offset), p.u, None) == 0
    torch.cuda.synchronize()
    a, b = one.cpu().numpy().view(np.uint32), many.cpu().numpy().view(np.uint32)
    np.testing.assert_array_equal(a, b)
