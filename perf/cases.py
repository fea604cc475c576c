"""Performance cases of the quantum-trajectory library: the calls its users make, over their real range of sizes.

Each case is a dict of plain values.  ``kind`` says which public entry points a pass goes through:

  run      ``Run`` on a fused circuit: whole noisy trajectories, densities and (small states) bitstrings
  apply    ``qt_state_apply``: a layer of fused gates on a caller-owned state
  measure  ``qt_state_reduced_density``, ``qt_state_kraus_probabilities`` (narrow channels),
           ``qt_state_expect_z`` and ``qt_state_sample`` on a caller-owned state
  channel  ``qt_state_kraus_probabilities`` of wide (4-6 qubit) channels
  batch    ``Batch.run``: one trajectory of each of many small circuits in one launch
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2111_02396_gb300 as qt
import qtsynth as qs


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # a user's first call: a 10-qubit noisy chain, a few trajectories with bitstrings and densities;
        # latency, launches and host round trips count
        dict(name="run_chain10", kind="run", rows=1, cols=10, depth=16, dep1=1e-3, dep2=1e-2, ad=1e-3, pd=0.0,
             fuse=2, traj=16, samples=100, tf32=False, share=False),
        # the noise-sweep size: 20 qubits, states that stay in cache, several trajectories
        dict(name="run_grid20", kind="run", rows=4, cols=5, depth=20, dep1=0.0, dep2=0.0, ad=5e-4, pd=5e-4,
             fuse=4, traj=8, samples=0, tf32=False, share=False),
        # the headline workload: one trajectory of the 30-qubit grid
        dict(name="run_grid30", kind="run", rows=5, cols=6, depth=20, dep1=0.0, dep2=0.0, ad=5e-4, pd=5e-4,
             fuse=4, traj=1, samples=0, tf32=False, share=False),
        # the precision option: 6-qubit fused gates in split TF32 on the 26-qubit grid of the error runs
        dict(name="run_tf32_grid26", kind="run", rows=2, cols=13, depth=24, dep1=1e-3, dep2=1e-3, ad=0.0, pd=0.0,
             fuse=6, traj=1, samples=0, tf32=True, share=False),
        # fused gates one by one on a caller's 28-qubit state: widths 1-4, low, middle, high and mixed targets
        dict(name="apply_k1to4_n28", kind="apply", n=28, tf32=False,
             gates="2,3,8,9 / 0,25,26,27 / 19,12,18,13 / 5,11,20 / 26,27 / 0"),
        # the widest fused gates in FP32
        dict(name="apply_k5k6_n27", kind="apply", n=27, tf32=False,
             gates="3,4,9,10,16 / 22,23,24,25,26 / 0,1,6,7,12,13 / 13,14,19,20,25,26"),
        # the same widths with the split-TF32 option, over the target patterns of grid circuits
        dict(name="apply_tf32_n28", kind="apply", n=28, tf32=True,
             gates="0,1,8,9,16 / 3,4,11,12,20 / 0,1,8,9,16,17 / 2,3,9,10,17,18 / 1,2,3,9,10,11 / 22,23,24,25,26,27"),
        # observables of a small state: every call is a few microseconds of device work
        dict(name="measure_n17", kind="measure", n=17, sets="4 / 0,16 / 3,9,11", terms=17, samples=100),
        # observables of a large state: each call reads 4 GiB
        dict(name="measure_n29", kind="measure", n=29, sets="28 / 5,6 / 0,1,17", terms=29, samples=1000),
        # branch probabilities of correlated noise on 4, 5 and 6 qubits
        dict(name="channel_n25", kind="channel", n=25, sets="2,3,8,9 / 12,4,11,5,19 / 0,6,12,18,23,24", ops="4 4 3"),
        # a batch of small circuits, 8-12 qubits: states in shared memory
        dict(name="batch_n8to12", kind="batch", circuits=50, repeats=32, nmin=8, nmax=12, depth=40, fuse=3, samples=100),
        # the batched workload's mix, 8-18 qubits, most of the work in states of global memory
        dict(name="batch_n8to18", kind="batch", circuits=55, repeats=12, nmin=8, nmax=18, depth=40, fuse=3, samples=100),
    ]


def _pick(rng, n, q):
    return rng.sample(range(n), q)


def _text(sets):
    return " / ".join(",".join(str(x) for x in s) for s in sets)


def draw(rng):
    kind = rng.choice(["run", "run", "apply", "apply", "measure", "channel", "batch"])
    if kind == "run":
        tf32 = rng.random() < 0.3
        chain = rng.random() < 0.4
        if tf32:
            rows, cols = rng.choice([(1, 17), (2, 9), (3, 7), (4, 6), (2, 13)])
        elif chain:
            rows, cols = 1, rng.randint(6, 22)
        else:
            rows, cols = rng.choice([(2, 4), (3, 3), (3, 4), (3, 5), (4, 4), (3, 6), (4, 5), (3, 7), (4, 6), (5, 5), (4, 7)])
        n = rows * cols
        depolar = rng.random() < 0.5
        p = 10.0 ** rng.uniform(-4.0, -2.5)
        # fewer trajectories of larger states
        traj = max(1, min(rng.randint(1, 24), 1 << max(0, 23 - n)))
        return dict(kind="run", rows=rows, cols=cols, depth=rng.randint(8, 24), dep1=p if depolar else 0.0,
                    dep2=2 * p if depolar else 0.0, ad=0.0 if depolar and tf32 else p, pd=0.0 if depolar else p,
                    fuse=rng.choice([5, 6]) if tf32 else rng.choice([2, 3, 4, 4]), traj=traj,
                    samples=rng.choice([0, 20, 100]) if n <= 10 else 0, tf32=tf32, share=rng.random() < 0.3)
    if kind == "apply":
        n = rng.randint(6, 29)
        tf32 = n >= 13 and rng.random() < 0.4
        widths = [rng.choice([5, 6]) if tf32 else rng.randint(1, 6 if n >= 13 else 5) for _ in range(rng.randint(1, 8))]
        return dict(kind="apply", n=n, tf32=tf32, gates=_text([_pick(rng, n, w) for w in widths]))
    if kind == "measure":
        n = rng.randint(6, 30)
        return dict(kind="measure", n=n, sets=_text([_pick(rng, n, rng.randint(1, 3)) for _ in range(rng.randint(1, 4))]),
                    terms=rng.randint(1, 40), samples=int(round(10.0 ** rng.uniform(0.0, 3.5))))
    if kind == "channel":
        n = rng.randint(6, 26)
        qs_ = [rng.randint(4, 6) for _ in range(rng.randint(1, 3))]
        return dict(kind="channel", n=n, sets=_text([_pick(rng, n, q) for q in qs_]),
                    ops=" ".join(str(rng.randint(2, 6)) for _ in qs_))
    nmax = rng.randint(8, 18)
    return dict(kind="batch", circuits=rng.randint(8, 48), repeats=rng.randint(1, 16 if nmax <= 14 else 6),
                nmin=rng.randint(6, nmax), nmax=nmax, depth=rng.randint(8, 40), fuse=rng.choice([2, 3, 3, 4]),
                samples=rng.choice([10, 33, 100]))


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _sets(text):
    return [[int(x) for x in part.split(",")] for part in text.split("/")]


def _unitary(d, rng):
    q, r = np.linalg.qr(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)))
    return q * (np.diag(r) / np.abs(np.diag(r)))[None, :]


def _kraus(d, m, rng):
    v = _unitary(d * m, rng)[:, :d]
    return np.stack([v[i * d:(i + 1) * d] for i in range(m)])


def _state(n, seed):
    """A random un-normalized state, as trajectories hold between flush points."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * seed + n)
    v = torch.randn(2 << n, generator=g, device="cuda", dtype=torch.float32)
    v.mul_(0.97 * 2.0 ** (-(n + 1) / 2))
    return torch.view_as_complex(v.view(-1, 2))


def _circuit(case, seed):
    noise = dict(dep1=case["dep1"] or None, dep2=case["dep2"] or None,
                 layer_ad=case["ad"] or None, layer_pd=case["pd"] or None)
    if case["rows"] == 1:
        return qs.chain_circuit(case["cols"], case["depth"], seed, **noise)
    return qs.grid_circuit(case["rows"], case["cols"], case["depth"], seed, **noise)


def _gate_mats(case, seed):
    rng = np.random.default_rng([11, seed])
    return [(s, _unitary(1 << len(s), rng)) for s in _sets(case["gates"])]


def _channels(case, seed):
    """(qubits, Kraus operators) per set; two random operators each unless the case gives the counts."""
    rng = np.random.default_rng([12, seed])
    sets = _sets(case["sets"])
    counts = [int(x) for x in case["ops"].split()] if "ops" in case else [2] * len(sets)
    return [(s, _kraus(1 << len(s), m, rng)) for s, m in zip(sets, counts)]


def _masks(n, terms, seed):
    """Single-qubit densities first, then random Z-strings."""
    rng = np.random.default_rng([13, seed])
    m = [1 << q for q in range(min(n, terms))]
    m += [int(x) for x in rng.integers(1, 1 << n, terms - len(m))]
    return np.array(m, dtype=np.uint64)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind == "run":
        circ = qt.Circuit.from_synth(_circuit(case, seed))
        st["fused"] = qt.Fused(circ, case["fuse"])
        st["masks"] = _masks(circ.num_qubits, circ.num_qubits, seed)
    elif kind == "batch":
        rng = np.random.default_rng([14, seed])
        span = case["nmax"] - case["nmin"] + 1
        circs = [qt.Circuit.from_synth(_batch_circuit(case["nmin"] + i % span, case["depth"], rng))
                 for i in range(case["circuits"])]
        fused = qt.fuse_many(circs, case["fuse"])
        st["batch"] = qt.Batch([f for f in fused for _ in range(case["repeats"])])
    else:
        st["psi"] = _state(case["n"], seed)
        if kind == "apply":
            st["gates"] = _gate_mats(case, seed)
            st["work"] = torch.empty_like(st["psi"])
        else:
            st["channels"] = _channels(case, seed)
            if kind == "measure":
                st["masks"] = _masks(case["n"], case["terms"], seed)
    return st


def _batch_circuit(n, depth, rng):
    """Chain circuit of the batched workload: depolarizing and amplitude damping 1e-3 per gate-qubit."""
    return qs.compact.layered_compact(n, depth, rng, lambda l: [(i, i + 1) for i in range(l % 2, n - 1, 2)],
                                      dep1=1e-3, dep2=1e-3, per_gate_ad=1e-3)


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def run(state):
    case, seed = state["case"], state["seed"]
    kind = case["kind"]
    if kind == "run":
        r = qt.Run(state["fused"], case["traj"], seed=seed, precision=qt.QT_TF32X3 if case["tf32"] else qt.QT_FP32,
                   samples_per_traj=case["samples"], z_masks=state["masks"], share_prefix=case["share"],
                   stream=_stream())
        kraus, stage = r.kraus_indices()
        return dict(expectation=r.expectation(), norms=r.norms(), samples=r.samples(), kraus=kraus, stage=stage)
    if kind == "batch":
        b = state["batch"].run(seed=seed, samples_per_traj=case["samples"], use_graph=True, stream=_stream())
        return b.samples()
    n, psi = case["n"], state["psi"]
    if kind == "apply":
        work = state["work"]
        work.copy_(psi)                      # the caller keeps its initial state
        for qubits, u in state["gates"]:
            qt.qt_state_apply(work.data_ptr(), n, qubits, u, precision=qt.QT_TF32X3 if case["tf32"] else qt.QT_FP32,
                              stream=_stream())
        return work
    ptr = psi.data_ptr()
    out = {}
    for i, (qubits, ks) in enumerate(state["channels"]):
        p, norm = qt.qt_state_kraus_probabilities(ptr, n, qubits, ks, stream=_stream())
        out[f"p{i}"], out[f"norm{i}"] = p, norm
        if kind == "measure":
            out[f"rho{i}"] = qt.qt_state_reduced_density(ptr, n, qubits, stream=_stream())
    if kind == "measure":
        out["z"] = qt.qt_state_expect_z(ptr, n, state["masks"], stream=_stream())
        out["samples"] = qt.qt_state_sample(ptr, n, seed, 0, case["samples"], stream=_stream())
    return out


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "run":
        # a state too large for the chip is written and read at least once per trajectory; every rotation
        # is a 2x2 product per amplitude pair (16 flops per amplitude), CZ and damping factors not counted
        n = case["rows"] * case["cols"]
        amps = float(1 << n) * case["traj"]
        return {"bytes": 16.0 * amps, "flops": (16.0 * n * case["depth"] + 3.0) * amps}
    if kind == "batch":
        # the states fit the chip or its cache; the samples go out
        n = 0.5 * (case["nmin"] + case["nmax"])
        count = case["circuits"] * case["repeats"]
        amps = sum(2.0 ** x for x in range(case["nmin"], case["nmax"] + 1)) / (case["nmax"] - case["nmin"] + 1)
        return {"bytes": 8.0 * count * case["samples"], "flops": count * amps * 16.0 * n * case["depth"]}
    amps = float(1 << case["n"])
    if kind == "apply":
        # each call reads and writes the caller's state; so does the copy
        widths = [len(s) for s in _sets(case["gates"])]
        return {"bytes": 16.0 * amps * (1 + len(widths)), "flops": amps * sum(2.0 ** (w + 3) for w in widths)}
    # each call reads the state once; a 2^q x 2^q density costs 4 * 2^q multiply-adds per amplitude, half of
    # them by symmetry
    widths = [len(s) for s in _sets(case["sets"])]
    flops = amps * sum(4.0 * 2.0 ** w for w in widths)
    if kind == "channel":
        return {"bytes": 8.0 * amps * len(widths), "flops": flops}
    passes = 2 * len(widths) + -(-case["terms"] // 16) + 1
    return {"bytes": 8.0 * amps * passes, "flops": 2 * flops + amps * (6.0 + case["terms"] / 8.0)}


# ----------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ----------------------------------------------------------------------------
def _split(psi, qubits):
    """psi as [2^q, rest] with index bit b of the first axis = qubits[b], and the way back."""
    n = int(math.log2(psi.numel()))
    order = sorted(qubits, reverse=True)
    shape, at = [], n
    for q in order:
        shape += [1 << (at - 1 - q), 2]
        at = q
    shape.append(1 << at)
    axis = {q: 2 * i + 1 for i, q in enumerate(order)}
    front = [axis[q] for q in reversed(qubits)]
    perm = front + [i for i in range(len(shape)) if i not in front]
    v = psi.view(shape).permute(perm)
    inverse = [perm.index(i) for i in range(len(perm))]
    return v.reshape(1 << len(qubits), -1), list(v.shape), inverse


def _apply64(psi, qubits, u):
    q = len(qubits)
    if q == 1:
        v = psi.view(-1, 2, 1 << qubits[0])
        if u[0, 1] == 0 and u[1, 0] == 0:
            if u[0, 0] != 1:
                v[:, 0] *= complex(u[0, 0])
            if u[1, 1] != 1:
                v[:, 1] *= complex(u[1, 1])
            return psi
        a = v[:, 0].clone()
        b = v[:, 1].clone()
        v[:, 0] = complex(u[0, 0]) * a + complex(u[0, 1]) * b
        v[:, 1] = complex(u[1, 0]) * a + complex(u[1, 1]) * b
        return psi
    if q == 2 and np.count_nonzero(u - np.diag(np.diag(u))) == 0:
        lo, hi = sorted(qubits)
        v = psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
        for i in range(4):
            f = complex(u[i, i])
            bits = {qubits[0]: i & 1, qubits[1]: i >> 1}
            if f != 1:
                v[:, bits[hi], :, bits[lo]] *= f
        return psi
    rows, shape, inverse = _split(psi, qubits)
    out = torch.tensor(u, dtype=torch.complex128, device=psi.device) @ rows
    return out.view(shape).permute(inverse).reshape(-1)


def _rho64(psi, qubits):
    rows, _, _ = _split(psi, qubits)
    return (rows @ rows.conj().T).cpu().numpy()


def _z64(psi, masks):
    n = int(math.log2(psi.numel()))
    w = psi.real ** 2 + psi.imag ** 2
    total = w.sum()
    out = []
    for m in masks:
        m, v = int(m), w
        for q in range(n - 1, -1, -1):       # fold the highest qubit into the sum or the difference of its halves
            a, b = v.view(2, -1)
            v = a - b if (m >> q) & 1 else a + b
        out.append(float(v[0] / total))
    return np.array(out)


def _uniform(seed, traj, stream, index):
    """Philox4x32-10 (Salmon et al. 2011) of counter (traj, stream, index): a uniform of 53 bits."""
    c = [traj & 0xFFFFFFFF, traj >> 32, stream, index]
    k = [seed & 0xFFFFFFFF, seed >> 32]
    for _ in range(10):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [(b >> 32) ^ c[1] ^ k[0], b & 0xFFFFFFFF, (a >> 32) ^ c[3] ^ k[1], a & 0xFFFFFFFF]
        k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
    return (((c[0] >> 5) << 26) | (c[1] >> 6)) * 2.0 ** -53


def _trajectory64(circ, seed, traj):
    """One trajectory with delayed inner products: lower bounds first, probabilities where they do not decide."""
    psi = torch.zeros(1 << circ.num_qubits, dtype=torch.complex128, device="cuda")
    psi[0] = 1.0
    channel = 0
    for op in circ.ops:
        qubits = list(op.qubits)
        if op.kind == qs.KIND_GATE:
            psi = _apply64(psi, qubits, op.mats[0])
            continue
        r = _uniform(seed, traj, 0, channel)
        channel += 1
        mix = op.kind == qs.KIND_MIXTURE
        if mix:
            bound = op.probs / op.probs.sum()
        else:
            bound = [max(np.linalg.eigvalsh(k.conj().T @ k)[0], 0.0) for k in op.mats]
        pick = None
        for i, p in enumerate(bound):
            if r < p:
                pick = op.mats[i]
                break
            r -= p
        if pick is None:
            rho = _rho64(psi, qubits)
            norm = np.trace(rho).real
            ks = [math.sqrt(p) * k for p, k in zip(bound, op.mats)] if mix else list(op.mats)
            ps = [np.trace(k.conj().T @ k @ rho).real for k in ks]
            for k, p, low in zip(ks, ps, bound):
                width = max(p / norm - low, 0.0)
                if width > 0.0:
                    pick = k / math.sqrt(p)
                if r < width:
                    break
                r -= width
        psi = _apply64(psi, qubits, pick)
    return psi


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return None                          # samples: whole numbers
    if kind == "run":
        n = case["rows"] * case["cols"]
        if n > 26 or float(1 << n) * case["traj"] > 1 << 26:
            return None
        circ = _circuit(case, seed)
        masks = _masks(n, n, seed)
        z, norms = [], []
        for t in range(case["traj"]):
            psi = _trajectory64(circ, seed, t)
            norms.append(float((psi.real ** 2 + psi.imag ** 2).sum()))
            z.append(_z64(psi, masks))
        return dict(expectation=np.array(z), norms=np.array(norms), samples=None, kraus=None, stage=None)
    psi = _state(case["n"], seed).to(torch.complex128)
    if kind == "apply":
        for qubits, u in _gate_mats(case, seed):
            psi = _apply64(psi, qubits, u)
        return psi
    out = {}
    for i, (qubits, ks) in enumerate(_channels(case, seed)):
        rho = _rho64(psi, qubits)
        out[f"p{i}"] = np.array([np.trace(k.conj().T @ k @ rho).real for k in ks])
        out[f"norm{i}"] = float(np.trace(rho).real)
        if kind == "measure":
            out[f"rho{i}"] = rho
    if kind == "measure":
        out["z"] = _z64(psi, _masks(case["n"], case["terms"], seed))
        out["samples"] = None
    return out
