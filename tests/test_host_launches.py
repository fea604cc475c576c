"""Host code around the launches, on the CPU: libqt.so on a CUDA runtime that records kernels
instead of running them (fake_cudart.cpp, preloaded into a child process)."""
import os
import subprocess
import sys
import textwrap

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PRELUDE = """
import ctypes, os
import numpy as np
import paper_2111_02396_gb300 as qt
import qtsynth as qs
from paper_2111_02396_gb300.qt import QtError
fake = ctypes.CDLL(os.environ["LD_PRELOAD"])
fake.fake_launches.restype = ctypes.c_char_p
fake.fake_fail_alloc.argtypes = [ctypes.c_size_t, ctypes.c_int]
qt.load()

def launches(part=""):
    rows = [x.split() for x in fake.fake_launches().decode().splitlines()]
    return [(name, int(g), int(b), int(s)) for name, g, b, s in rows if part in name]
"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    from paper_2111_02396_gb300 import build
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I", os.path.join(CUDA, "include"),
                    os.path.join(HERE, "fake_cudart.cpp"), "-o", so], check=True)

    def run(code):
        env = dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT)
        r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(code)], env=env, cwd=ROOT,
                           capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout + r.stderr

    return run


@pytest.mark.parametrize("k", [3, 4, 6])
@pytest.mark.parametrize("n", [9, 14])
def test_batch_shared_memory_with_empty_circuits(child, k, n):
    """The matrix buffers of a class are sized for its widest gate: an empty circuit, which has the
    same first gate as the circuit packed after it, takes nothing from them."""
    child(f"""
    n, k = {n}, {k}
    real = [qt.Fused(qt.Circuit.from_synth(qs.chain_circuit(n, 8, s, dep1=1e-2)), k) for s in (1, 2)]
    empty = [qt.Fused(qt.Circuit.from_synth(qs.Circuit(m)), k) for m in (n, 2, 20)]
    w = max(len(f.gate(g)["targets"]) for f in real for g in range(f.info()["num_fused"]))
    assert w == k
    narrow = min(w, 4)
    need = 8 * ((1 << n) + (2 << 2 * narrow) + ((1 << 2 * w) if w > 4 else 0))
    cls = "k_batch_smemILi512E" if n == 14 else "k_batch_smemILi128E"
    for batch in (real, [empty[0]] + real, [empty[1], real[0], empty[0], real[1], real[0]], empty + real + empty):
        fake.fake_clear()
        qt.Batch(batch).run(seed=1)
        got = [x[3] for x in launches(cls)]
        assert got == [need], (batch, got, need)
    """)


@pytest.mark.parametrize("kernel,call", [
    ("k_rdmILi1", "qt.qt_state_reduced_density(p, 12, [3])"),
    ("k_rdmILi2", "qt.qt_state_reduced_density(p, 12, [0, 3])"),
    ("k_rdm3", "qt.qt_state_reduced_density(p, 12, [5, 0, 3])"),
    ("k_rdmILi2", "qt.qt_state_kraus_probabilities(p, 12, [7, 3], K(2))"),
    ("k_kraus_normsILi4", "qt.qt_state_kraus_probabilities(p, 12, [7, 3, 1, 2], K(4))"),
    ("k_norms64", "qt.qt_state_kraus_probabilities(p, 12, [7, 3, 1, 2, 4, 5], K(6))"),
    ("k_gramILi4", "qt.qt_state_kraus_probabilities(p, 22, [7, 3, 1, 2], K(4))"),
    ("k_gram_matrix", "qt.qt_state_kraus_probabilities(p, 23, [7, 3, 1, 2, 4], K(5))"),
    ("k_kraus_trace", "qt.qt_state_kraus_probabilities(p, 22, [7, 3, 1, 2], K(4))"),
    ("k_expect", "qt.qt_state_expect_z(p, 8, [1, 3])"),
    ("k_expect_wht", "qt.qt_state_expect_z(p, 12, [1, 3])"),
    ("k_finalize", "qt.qt_state_expect_z(p, 12, [1, 3])"),
    ("k_cdf_sub", "qt.qt_state_sample(p, 12, 1, 0, 10)"),
    ("k_cdf_blk", "qt.qt_state_sample(p, 12, 1, 0, 10)"),
    ("k_cdf_scan", "qt.qt_state_sample(p, 12, 1, 0, 10)"),
    ("k_sample", "qt.qt_state_sample(p, 12, 1, 0, 10)"),
    ("k_apply", "qt.qt_state_apply(p, 12, [3, 1], np.eye(4))"),
    ("k_batch_glob", "batch.run(seed=1)"),
    ("k_batch_smem", "batch.run(seed=1)"),
])
def test_failed_launch_is_reported(child, kernel, call):
    """A launch that the runtime refuses ends the call with an error, also where a dependent launch
    follows it, and leaves nothing behind for the next call."""
    child(f"""
    K = lambda q: np.eye(1 << q)[None]
    buf = np.zeros(1 << 16, np.complex64)
    p = (buf.ctypes.data + 255) & ~255
    batch = qt.Batch([qt.Fused(qt.Circuit.from_synth(qs.chain_circuit(n, 4, 1, dep1=1e-2)), 3) for n in (9, 16)])
    call = lambda: {call}
    call()
    assert launches("{kernel}")
    fake.fake_fail(b"{kernel}")
    try:
        call()
    except QtError as e:
        assert e.status == qt.qt.QT_ERR_CUDA
    else:
        raise AssertionError("the call returned a result")
    fake.fake_fail(b"")
    call()
    """)


@pytest.mark.parametrize("flushes,share,keep", [(False, False, False), (True, False, True), (True, True, False)])
def test_timeout_flag_ends_a_run(child, flushes, share, keep):
    """A tensor-core wait that ran out ends a run at the next stage-2 choice, or at the latest with the
    eighth trajectory."""
    child(f"""
    n, T = 13, 40
    c = qs.Circuit(n)
    rng = np.random.default_rng(1)
    for m in range(0, 12, 2):
        q = sorted(int(x) for x in rng.choice(n, 6, replace=False))
        c.gate(np.linalg.qr(rng.normal(size=(64, 64)) + 1j * rng.normal(size=(64, 64)))[0], tuple(q), m)
        if {flushes}:
            c.channel(qs.amplitude_damping(0.9), (q[0],), m + 1)
    f = qt.Fused(qt.Circuit.from_synth(c), 6)
    run = lambda t: qt.Run(f, t, seed=3, precision=qt.QT_TF32X3, share_prefix={share}, keep_states={keep})
    run(1)
    one = len(launches("k_apply_tc"))
    fake.fake_clear()
    st = run(T).stats()
    assert len(launches("k_apply_tc")) > T
    assert (st["prob_passes"] > 0) == {flushes}
    fake.fake_clear()
    fake.fake_set(b"k_apply_tc")
    for t in (1, T):
        try:
            run(t)
        except QtError as e:
            assert e.status == qt.qt.QT_ERR_TIMEOUT
        else:
            raise AssertionError("the run returned")
    got = len(launches("k_apply_tc"))                        # of t = 1 and of T
    assert one > 2 and got <= (2 if {flushes} else 9) * one, (one, got)
    fake.fake_set(b"")
    run(2)
    """)


@pytest.mark.parametrize("sizes,distinct", [((8, 9, 10), 1), ((9, 11, 13), 2), ((9, 14), 3), ((15, 16), 2)])
def test_autotuner_times_each_launch_once(child, sizes, distinct):
    """Values of `threads` that launch the same CTAs are one choice, the largest of them: equal times
    are not left to noise, which would pick how sums are split."""
    child(f"""
    cs = [qt.Circuit.from_synth(qs.chain_circuit(n, 3, n, dep1=1e-2)) for n in {sizes}]
    best, table = qt.autotune_batch(cs, kmin=2, kmax=3)
    cls = "global" if {sizes}[0] > 14 else "shared"
    rows = [[table[(cls, k, t)] for t in (128, 256, 512)] for k in (2, 3)]
    assert all(t > 0 for r in rows for t in r)
    one = [x[2] for x in launches("k_batch")]
    # 2 widths, {distinct} values, 3 runs of a launch for each class present
    classes = len(set(14 if n == 14 else 13 if n == 13 else 12 if n > 10 else 10 for n in {sizes} if n <= 14)) or 1
    assert len(one) == 2 * {distinct} * 3 * classes, (len(one), classes)
    assert best["threads_" + cls] == 512            # every run takes 1 ms here: the first that was timed
    """)


def test_lane_after_an_allocation_failure(child):
    """The batch lane keeps its buffers between launches; a request that is deferred because they could
    not grow is launched with buffers of its size."""
    child("""
    f = qt.Fused(qt.Circuit.from_synth(qs.chain_circuit(9, 6, 1, dep1=1e-2)), 3)
    srv = qt.Server(1 << 33, max_slots=1, small_n_max=14)
    for samples, fails in ((10, 0), (4000, 1), (16000, 2)):
        fake.fake_clear()
        fake.fake_fail_alloc(64 * samples * 8, fails)
        i = srv.submit(f, seed=1, num_traj=64, samples_per_traj=samples)
        srv.wait(i, timeout_s=60)
        smp, inf = srv.result(i)
        assert smp.shape == (64, samples) and not smp.any()
        assert len(launches("k_batch_smem")) == 1
    srv.close()
    """)


@pytest.mark.parametrize("keep", [False, True])
def test_batch_after_an_allocation_failure(child, keep):
    """A run whose state arena cannot be had launches nothing, and neither does the next one."""
    child(f"""
    f = [qt.Fused(qt.Circuit.from_synth(qs.chain_circuit(n, 4, n, dep1=1e-2)), 3) for n in (16, 9)]
    b = qt.Batch(f)
    args = dict(seed=1, samples_per_traj=5, keep_states={keep})
    for first in (None, dict(seed=1, samples_per_traj=4)):
        if first:
            b.run(**first)                      # a layout that the next run replaces
        fake.fake_clear()
        fake.fake_fail_alloc(1 << 18, 2)
        for _ in range(2):
            try:
                b.run(**args)
            except QtError as e:
                assert e.status == qt.qt.QT_ERR_OUT_OF_MEMORY
            else:
                raise AssertionError("the run returned")
        assert not launches("k_batch")
        b.run(**args)
        assert len(launches("k_batch")) == 2
    """)
