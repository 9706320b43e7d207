"""Measured workloads of the state-vector simulator, through its public entry points.

Each case is a dict of plain values with a ``kind``:

``qpe``      phase estimation from |0...0> (``sv_reset`` + ``sv_apply_circuit``) and its
             measured bitstring (``sv_argmax`` over the counting register)
``random``   layers of U3 on every qubit and CZ on a random matching, from |0...0>: the
             amplitudes on the device
``general``  a dynamic circuit: single-qubit and controlled gates, Toffoli-like gates,
             two-qubit unitaries and mid-circuit measurements, one sv_apply_circuit call
``readout``  reading out a state that is already there: the marginals of a small and of a
             large register into device memory, and inverse-CDF samples of the large one
``batch``    many independent QPE instances in one launch (``sv_batch_run``)

A program keeps its handle (and its state buffer, a torch tensor) and runs one circuit
after another on it, so ``prepare`` makes the handle, the gate list and the read-out
requests, and ``run`` starts from |0...0> each time.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2605_15098_gb300 import circuits as C
from paper_2605_15098_gb300 import sv

DTYPES = {"c64": (sv.SV_C64, torch.complex64, 8), "c128": (sv.SV_C128, torch.complex128, 16)}
VIEW_QUBITS = 20  # QPE states up to this size are returned beside the bitstring


def listed():
    return [
        # a small instance in the library's default configuration: latency of a whole call
        {"name": "qpe_n11_c64", "kind": "qpe", "n": 11, "targets": 4, "dtype": "c64", "tuned": False},
        # an ordinary instance, default configuration
        {"name": "qpe_n20_c64", "kind": "qpe", "n": 20, "targets": 4, "dtype": "c64", "tuned": False},
        # the headline benchmark: 28 qubits in the configuration the autotuner picks for it
        {"name": "qpe_n28_c64", "kind": "qpe", "n": 28, "targets": 4, "dtype": "c64", "tuned": True},
        # double precision phase estimation
        {"name": "qpe_n24_c128", "kind": "qpe", "n": 24, "targets": 4, "dtype": "c128", "tuned": False},
        # random circuits: a small state, an odd ordinary one, a deep one, the largest
        {"name": "random_n15_c64", "kind": "random", "n": 15, "depth": 20, "dtype": "c64"},
        {"name": "random_n19_c64", "kind": "random", "n": 19, "depth": 20, "dtype": "c64"},
        {"name": "random_n25_c64", "kind": "random", "n": 25, "depth": 20, "dtype": "c64"},
        {"name": "random_n28_c64", "kind": "random", "n": 28, "depth": 8, "dtype": "c64"},
        # random circuit in double precision
        {"name": "random_n21_c128", "kind": "random", "n": 21, "depth": 10, "dtype": "c128"},
        # a dynamic circuit with every general gate kind
        {"name": "general_n23_c64", "kind": "general", "n": 23, "depth": 6, "dtype": "c64"},
        # a few ancilla qubits and a 20-qubit register read from a 26-qubit state
        {"name": "readout_n26_c64", "kind": "readout", "n": 26, "small": 3, "large": 20, "shots": 4096,
         "dtype": "c64"},
        # a batch of QPE instances of mixed sizes
        {"name": "batch_512", "kind": "batch", "count": 512, "n_lo": 10, "n_hi": 20},
    ]


def draw(rng: random.Random):
    kind = rng.choice(["qpe", "qpe", "random", "random", "random", "general", "readout", "batch"])
    dtype = rng.choice(["c64", "c64", "c128"])
    if kind == "qpe":
        n = rng.randint(8, 27 if dtype == "c64" else 23)
        tuned = dtype == "c64" and n >= 22 and rng.random() < 0.7
        return {"kind": kind, "n": n, "targets": rng.randint(1, 6), "dtype": dtype, "tuned": tuned}
    if kind == "random":
        n = rng.randint(8, 28 if dtype == "c64" else 22)
        top = 40 if n <= 24 else 8  # a drawn circuit costs no more than the listed ones
        if dtype == "c128":
            top = 20 if n <= 20 else 6
        return {"kind": kind, "n": n, "depth": rng.randint(3, top), "dtype": dtype}
    if kind == "general":
        return {"kind": kind, "n": rng.randint(8, 24 if dtype == "c64" else 21), "depth": rng.randint(3, 8),
                "dtype": dtype}
    if kind == "readout":
        n = rng.randint(10, 27 if dtype == "c64" else 26)
        return {"kind": kind, "n": n, "small": rng.randint(1, 8), "large": rng.randint(8, min(n, 22)),
                "shots": int(2 ** rng.uniform(0, 14)), "dtype": dtype}
    hi = rng.randint(12, 20)
    return {"kind": kind, "count": int(2 ** rng.uniform(4, 9)), "n_lo": rng.randint(8, hi), "n_hi": hi}


# ---- inputs -----------------------------------------------------------------
def _general_circuit(n: int, depth: int, seed: int):
    """Seeded dynamic circuit: (gate array, number of measurements)."""
    r = random.Random(seed)
    g = np.random.RandomState(seed & 0x7FFFFFFF)
    recs, nmeas = [C.h(q) for q in range(n)], 0

    def haar(k):
        z = g.normal(size=(k, k)) + 1j * g.normal(size=(k, k))
        q, t = np.linalg.qr(z)
        d = np.diag(t)
        return q * (d / np.abs(d))

    for layer in range(depth):
        perm = list(range(n))
        r.shuffle(perm)
        for q in perm[: n // 2]:
            recs.append(C.u3(q, *(r.uniform(0.0, 2.0 * math.pi) for _ in range(3))))
        for a, b in zip(perm[0::4], perm[1::4]):
            recs.append(C.cp(a, b, r.uniform(-math.pi, math.pi)))
        for a, b in zip(perm[2::4], perm[3::4]):
            recs.append(C.cu(a, b, [[0, 1], [1, 0]]) if r.random() < 0.5 else C.cu(a, b, haar(2)))
        recs.append(C.swap(perm[0], perm[-1]))
        recs.append(C.mcu(r.sample(perm[1:], 2), perm[0], [[0, 1], [1, 0]]))
        recs += C.u2q(perm[1], perm[-2], haar(4))
        if layer % 3 == 1:  # far from both certain outcomes: no outcome sits on a CDF boundary
            recs.append(C.measure(perm[2], r.choice([0.07, 0.93])))
            nmeas += 1
    return C.gates(recs), nmeas


def _readout_request(case, seed):
    r = random.Random(seed)
    qs = list(range(case["n"]))
    small = r.sample(qs, min(case["small"], case["n"]))
    large = r.sample(qs, min(case["large"], case["n"]))
    u = np.random.RandomState(seed & 0x7FFFFFFF).random_sample(case["shots"])
    return sum(1 << q for q in small), sum(1 << q for q in large), u


def _random_state(case, seed, device="cuda"):
    """Normalised complex Gaussian amplitudes: the output statistics of a random circuit."""
    gen = torch.Generator(device=device).manual_seed(int(seed))
    _, dt, _ = DTYPES[case["dtype"]]
    t = torch.randn(1 << case["n"], dtype=dt, device=device, generator=gen)
    t /= math.sqrt(float(1 << case["n"]))
    return t


def _qpe_seed(seed):
    return C.DEFAULT_SEED + 7919 * int(seed)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        insts = C.qpe_batch(case["count"], _qpe_seed(seed), case["n_lo"], case["n_hi"])
        b = sv.sv_batch_create([(n, g, mask) for n, g, mask, _ in insts])
        return {"kind": kind, "batch": _Batch(b), "count": case["count"]}
    n = case["n"]
    code, dt, _ = DTYPES[case["dtype"]]
    if kind == "readout":
        amps = torch.empty(1 << n, dtype=dt, device="cuda")
        s = sv.State(n, code, tensor=amps)
        sv.sv_info(s.h)  # the buffer is the state from here on
        amps.copy_(_random_state(case, seed))
        ms, ml, u = _readout_request(case, seed)
        ps = torch.empty(1 << bin(ms).count("1"), dtype=torch.float64, device="cuda")
        pl = torch.empty(1 << bin(ml).count("1"), dtype=torch.float64, device="cuda")
        return {"kind": kind, "state": s, "small": ms, "large": ml, "u": u, "ps": ps, "pl": pl}
    amps = torch.empty(1 << n, dtype=dt, device="cuda")
    s = sv.State(n, code, tensor=amps)
    st = {"kind": kind, "state": s, "amps": amps, "n": n, "cfg": None}
    if kind == "qpe":
        g, _, info = C.qpe(n, _qpe_seed(seed), case["targets"])
        st["mask"] = info["mask"]
        if case["tuned"]:
            st["cfg"] = sv.make_config(sv.SV_MODE_PARTITIONED, chunk_qubits=9, flags=sv.SV_FLAG_NARROW_FIRST)
    elif kind == "random":
        g = C.random_circuit(n, case["depth"], _qpe_seed(seed))
    else:
        g, _ = _general_circuit(n, case["depth"], seed)
    st["gates"] = g
    return st


class _Batch:
    """Owner of a batch handle."""

    def __init__(self, b):
        self.b = b

    def __del__(self):
        if self.b:
            sv.sv_batch_destroy(self.b)
            self.b = None


# ---- one pass ---------------------------------------------------------------
def _logical(st):
    """The state buffer seen in logical qubit order (a view, by the handle's qubit map)."""
    n, amps = st["n"], st["amps"]
    phys = sv.sv_qubit_map(st["state"].h)
    if phys == list(range(n)):
        return amps
    # dimension d of the view holds bit n-1-d of the amplitude index
    return amps.view([2] * n).permute([n - 1 - phys[n - 1 - d] for d in range(n)])


def run(st):
    kind = st["kind"]
    if kind == "batch":
        idx, p, _ = sv.sv_batch_run(st["batch"].b, st["count"])
        return {"idx": idx, "p": p}
    s = st["state"]
    if kind == "readout":
        sv.sv_probabilities_device(s.h, st["small"], st["ps"].data_ptr())
        sv.sv_probabilities_device(s.h, st["large"], st["pl"].data_ptr())
        out = s.sample(st["large"], st["u"])
        return {"small": st["ps"], "large": st["pl"], "samples": out.astype(np.int64)}
    s.reset()
    s.apply(st["gates"], st["cfg"])
    if kind == "qpe":
        idx, p = s.argmax(st["mask"])
        out = {"idx": idx, "p": p}
        if st["n"] <= VIEW_QUBITS:
            out["state"] = _logical(st)
        return out
    if kind == "general":
        return {"bits": s.measurements().astype(np.int64), "state": _logical(st)}
    return _logical(st)


# ---- what a pass cannot do without ------------------------------------------
def _circuit_flops(g, n):
    """Operations of the list applied gate by gate, on the amplitudes each gate changes."""
    size, f = float(1 << n), 0.0
    for kind, num in zip(g["kind"].tolist(), g["num"].tolist()):
        if kind == C.H:
            f += 4.0 * size  # (a + b, a - b), scaled
        elif kind in (C.P, C.PK):
            f += 6.0 * size / 2
        elif kind in (C.CP, C.CPK):
            f += 6.0 * size / 4
        elif kind == C.CZ:
            f += 2.0 * size / 4
        elif kind in (C.U3, C.U):
            f += 14.0 * size
        elif kind == C.CU:
            f += 14.0 * size / 2
        elif kind == C.MCU:
            f += 14.0 * size / (1 << bin(num).count("1"))
        elif kind == C.U2Q:
            f += 30.0 * size
        elif kind == C.MEASURE:
            f += 6.0 * size
    return f


def work(case):
    if case["kind"] == "batch":
        by = fl = 0.0
        for n, s in C.batch_specs(case["count"], _qpe_seed(0), case["n_lo"], case["n_hi"]):
            t = n - 4
            by += 96.0 * C.qpe_gate_count(n) + 8.0 * (1 << n)
            fl += (1 << n) * (8.0 * t + 1.5 * (4 * t + t * (t - 1) / 2) + 4.0)
        return {"bytes": by, "flops": fl}
    n = case["n"]
    amp = DTYPES[case["dtype"]][2]
    state = float(amp << n)
    if case["kind"] == "readout":
        k = 8.0 * ((1 << min(case["small"], n)) + (1 << min(case["large"], n)))
        return {"bytes": state + k + 16.0 * case["shots"], "flops": 4.0 * (1 << n)}
    if case["kind"] == "qpe":
        g, _, _ = C.qpe(n, targets=case["targets"])
        extra = 4.0 * (1 << n)  # the marginal of the counting register
    elif case["kind"] == "random":
        g, extra = C.random_circuit(n, case["depth"]), 0.0
    else:
        (g, _), extra = _general_circuit(n, case["depth"], 0), 0.0
    return {"bytes": state + 96.0 * g.size, "flops": _circuit_flops(g, n) + extra}


# ---- the same in 64 bits, by plain torch ------------------------------------
def _axes(v, qubits):
    """View of the state with one dimension of 2 per given qubit first (in the given order)."""
    n = v.numel().bit_length() - 1
    order = sorted(qubits, reverse=True)
    shape, at, top = [], {}, n
    for q in order:
        shape += [1 << (top - q - 1), 2]
        at[q] = len(shape) - 1
        top = q
    shape.append(1 << top)
    w = v.view(shape)
    return w.permute([at[q] for q in qubits] + [i for i in range(len(shape)) if i not in at.values()])


def _apply2(v, t, m, controls=()):
    w = _axes(v, list(controls) + [t])[(1,) * len(controls)]
    a, b = w[0], w[1]
    na = m[0][0] * a + m[0][1] * b
    b.copy_(m[1][0] * a + m[1][1] * b)
    a.copy_(na)


def _simulate(n, gates):
    """Amplitudes (complex128, logical order) and measured bits of a gate list from |0...0>."""
    v = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    v[0] = 1.0
    bits, i = [], 0
    while i < len(gates):
        r = gates[i]
        k, t, c = int(r["kind"]), int(r["target"]), int(r["control"])
        p = [float(x) for x in r["p"]]
        mat = [[complex(p[0], p[1]), complex(p[2], p[3])], [complex(p[4], p[5]), complex(p[6], p[7])]]
        if k == C.X:
            _apply2(v, t, [[0, 1], [1, 0]])
        elif k == C.H:
            s = math.sqrt(0.5)
            _apply2(v, t, [[s, s], [s, -s]])
        elif k in (C.P, C.CP, C.CZ, C.PK, C.CPK):
            if k in (C.P, C.CP):
                ph = p[0]
            elif k == C.CZ:
                ph = math.pi
            else:
                den = 1 << int(r["log2den"])
                ph = 2.0 * math.pi * ((int(r["num"]) % den) / den)
            qs = [t] if k in (C.P, C.PK) else [c, t]
            f = -1.0 if k == C.CZ else complex(math.cos(ph), math.sin(ph))
            _axes(v, qs)[(1,) * len(qs)].mul_(f)
        elif k == C.SWAP:
            w = _axes(v, [t, c])
            tmp = w[0, 1].clone()
            w[0, 1].copy_(w[1, 0])
            w[1, 0].copy_(tmp)
        elif k == C.U3:
            a, b, d = p[0], p[1], p[2]
            e = lambda x: complex(math.cos(x), math.sin(x))  # noqa: E731
            _apply2(v, t, [[math.cos(a / 2), -e(d) * math.sin(a / 2)],
                           [e(b) * math.sin(a / 2), e(b + d) * math.cos(a / 2)]])
        elif k == C.U:
            _apply2(v, t, mat)
        elif k == C.CU:
            _apply2(v, t, mat, [c])
        elif k == C.MCU:
            _apply2(v, t, mat, [q for q in range(n) if (int(r["num"]) >> q) & 1])
        elif k == C.U2Q:
            rows = [[complex(gates[i + j]["p"][2 * e], gates[i + j]["p"][2 * e + 1]) for e in range(4)]
                    for j in range(4)]
            w = _axes(v, [c, t])  # [bit of control][bit of target]
            old = [w[e >> 1, e & 1].clone() for e in range(4)]
            for j in range(4):
                w[j >> 1, j & 1].copy_(sum(rows[j][e] * old[e] for e in range(4)))
            i += 3
        elif k == C.MEASURE:
            w = _axes(v, [t])
            p0, p1 = (float(torch.view_as_real(w[e].contiguous()).square().sum()) for e in range(2))
            out = 0 if p0 > p[0] * (p0 + p1) else 1
            w[1 - out].zero_()
            w[out].mul_(1.0 / math.sqrt(p1 if out else p0))
            bits.append(out)
        else:
            raise ValueError(k)
        i += 1
    return v, np.array(bits, dtype=np.int64)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        insts = C.qpe_batch(case["count"], _qpe_seed(seed), case["n_lo"], case["n_hi"])
        return {"idx": np.array([y for _, _, _, y in insts], dtype=np.uint64),
                "p": np.ones(len(insts), dtype=np.float64)}
    n = case["n"]
    if kind == "readout":
        v = _random_state(case, seed).to(torch.complex128)
        p = torch.view_as_real(v).square().sum(-1)
        ms, ml, _ = _readout_request(case, seed)
        out = []
        for mask in (ms, ml):
            qs = [q for q in range(n - 1, -1, -1) if (mask >> q) & 1]
            w = p
            # sum the other qubits out from the top down, so that the rest keeps its order
            left = list(range(n))
            for q in range(n - 1, -1, -1):
                if (mask >> q) & 1:
                    continue
                at = left.index(q)
                w = w.reshape(-1, 2, 1 << at).sum(1).reshape(-1)
                left.remove(q)
            assert len(left) == len(qs)
            out.append(w / w.sum())
        return {"small": out[0], "large": out[1], "samples": None}
    if kind == "qpe":
        g, _, info = C.qpe(n, _qpe_seed(seed), case["targets"])
        out = {"idx": info["y"], "p": 1.0}
        if n <= VIEW_QUBITS:
            out["state"] = _simulate(n, g)[0]
        return out
    if kind == "random":
        return _simulate(n, C.random_circuit(n, case["depth"], _qpe_seed(seed)))[0]
    g, _ = _general_circuit(n, case["depth"], seed)
    v, bits = _simulate(n, g)
    return {"bits": bits, "state": v}
