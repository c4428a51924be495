"""Timing cases: the work a user of this library has it do, through its public entry points.

A case names a kind of call, a qubit count, a dtype and the kind's own sizes; its circuit's structure depends on the
case alone, its angles, matrices and input state on the seed.  Kinds:

  gates      one lqs_apply_gate call per gate (gate by gate simulation; the single-gate sweeps)
  ansatz     |0..0> through the RY + RZ + CNOT-ladder ansatz on the fused path (a variational forward pass)
  qft        a state through the quantum Fourier transform with its final swaps
  universal  a state through N layers of phase gates and CNOT ladders
  windows    a state through runs of dense two-qubit unitaries, each run inside five neighbouring qubits
  expval     the transverse-field Ising energy of a state, with every word's value
  gradient   one variational step: forward, energy, adjoint gradient
  batch      forward, energy and gradient of many small circuits of uneven sizes in one call
"""
import math
import random
from collections import namedtuple

import numpy as np
import torch

import paper_2508_13615_gb300 as L

Op = namedtuple("Op", "name wires pidx matrix inverse", defaults=(-1, None, False))
Word = namedtuple("Word", "coeff x_mask z_mask")
Circuit = namedtuple("Circuit", "n_qubits ops params")

AMP = {"c64": 8, "c128": 16}
TORCH = {"c64": torch.complex64, "c128": torch.complex128}


def listed():
    return [
        # the 12-qubit single-gate suite: every gate on every target and ordered pair; launches and host calls count
        {"name": "gates12_c128", "kind": "gates", "n": 12, "dtype": "c128", "suite": True},
        # a gate-by-gate run on a large state: H, RZ, CNOT and a dense two-qubit gate on low, middle and high qubits
        {"name": "gates28_c128", "kind": "gates", "n": 28, "dtype": "c128", "suite": False},
        # a variational loop on one small circuit: forward, energy and gradient; latency counts
        {"name": "gradient14_c128", "kind": "gradient", "n": 14, "dtype": "c128", "layers": 4},
        # the headline circuit: 10 layers at 30 qubits, 16 GiB of complex128
        {"name": "ansatz30_c128", "kind": "ansatz", "n": 30, "dtype": "c128", "layers": 10},
        # the same family in single precision, at an odd qubit count and depth
        {"name": "ansatz29_c64", "kind": "ansatz", "n": 29, "dtype": "c64", "layers": 7},
        # the Fourier transform of a full state
        {"name": "qft29_c128", "kind": "qft", "n": 29, "dtype": "c128"},
        # the universal circuit: few operations per gate, long CNOT ladders (24 qubits: a state larger than L2)
        {"name": "universal24_c128", "kind": "universal", "n": 24, "dtype": "c128"},
        # dense two-qubit runs inside five-qubit windows: the tensor-core blocks
        {"name": "windows27_c64", "kind": "windows", "n": 27, "dtype": "c64", "windows": 6, "gates": 10},
        # measuring an energy of a large state
        {"name": "expval28_c128", "kind": "expval", "n": 28, "dtype": "c128"},
        # variational training at 24 qubits, 384 parameters
        {"name": "gradient24_c128", "kind": "gradient", "n": 24, "dtype": "c128", "layers": 8},
        # the same in single precision, at an odd qubit count
        {"name": "gradient23_c64", "kind": "gradient", "n": 23, "dtype": "c64", "layers": 8},
        # the serving load: 256 circuits of 10 to 20 qubits and 4 to 12 layers, with gradients
        {"name": "batch256_c64", "kind": "batch", "dtype": "c64", "count": 256, "n_min": 10, "n_max": 20},
    ]


def draw(rng):
    kind = rng.choice(["gates", "ansatz", "qft", "universal", "windows", "expval", "gradient", "gradient", "batch"])
    c = {"kind": kind, "dtype": rng.choice(["c64", "c128"])}
    if kind == "gates":
        c.update(n=rng.randint(8, 28), suite=False)
    elif kind == "ansatz":
        c.update(n=rng.randint(16, 29), layers=rng.randint(2, 10))
    elif kind == "qft":
        c.update(n=rng.randint(14, 29))
    elif kind == "universal":
        c.update(n=rng.randint(14, 24))
    elif kind == "windows":
        c.update(n=rng.randint(14, 27), windows=rng.randint(1, 6), gates=rng.randint(4, 12))
    elif kind == "expval":
        c.update(n=rng.randint(14, 28))
    elif kind == "gradient":
        c.update(n=rng.randint(6, 24), layers=rng.randint(2, 8))
    else:
        c.update(count=int(round(16 * 2 ** rng.uniform(0, 4))), n_min=rng.randint(6, 12), n_max=rng.randint(14, 20))
    return c


# ---------------------------------------------------------------------------
# circuits and observables
# ---------------------------------------------------------------------------

def ansatz_ops(n, layers):
    ops = []
    for l in range(layers):
        ops += [Op("RY", (q,), 2 * n * l + q) for q in range(n)]
        ops += [Op("RZ", (q,), 2 * n * l + n + q) for q in range(n)]
        ops += [Op("CNOT", (q, q + 1)) for q in range(n - 1)]
    return ops


def qft_circuit(n):
    ops, vals = [], []
    for j in range(n - 1, -1, -1):
        ops.append(Op("H", (j,)))
        for k in range(j - 1, -1, -1):
            ops.append(Op("ControlledPhaseShift", (k, j), len(vals)))
            vals.append(math.pi / 2.0 ** (j - k))
    ops += [Op("SWAP", (i, n - 1 - i)) for i in range(n // 2)]
    return Circuit(n, ops, np.array(vals))


def universal_angle(layer, q, n):
    return math.pi / 2.0 ** (1 + (layer + q) % n)


def universal_circuit(n):
    ops, vals = [], []
    for layer in range(n + 1):
        for q in range(n):
            ops.append(Op("PhaseShift", (q,), len(vals)))
            vals.append(universal_angle(layer, q, n))
        if layer < n:
            ops += [Op("CNOT", (q, q + 1)) for q in range(n - 1)]
    return Circuit(n, ops, np.array(vals))


def haar(dim, count, seed):
    r = np.random.default_rng(seed)
    z = r.standard_normal((count, dim, dim)) + 1j * r.standard_normal((count, dim, dim))
    q, t = np.linalg.qr(z)
    d = np.diagonal(t, axis1=1, axis2=2)
    return q * (d / np.abs(d))[:, None, :]


def window_wires(case):
    """The runs' gates: pairs of qubits inside windows spread over the register, the first at qubit 0."""
    n, w = case["n"], case["windows"]
    r = random.Random(97 * n + w)
    wires = []
    for i in range(w):
        s = (n - 5) * i // max(w - 1, 1)
        for _ in range(case["gates"]):
            wires.append(tuple(s + x for x in r.sample(range(5), 2)))
    return wires


def window_ops(case, seed):
    wires = window_wires(case)
    return [Op("U4", w, -1, u) for w, u in zip(wires, haar(4, len(wires), seed))]


def tfim(n):
    return [Word(1.0, 0, 3 << i) for i in range(n - 1)] + [Word(0.5, 1 << i, 0) for i in range(n)]


def gate_calls(case, seed):
    """(gate, wires, parameters or matrix) of each call."""
    n, r = case["n"], np.random.default_rng(seed)
    ang = lambda: [float(r.uniform(0, 2 * math.pi))]  # noqa: E731
    if case["suite"]:
        us = haar(2, n, seed + 1)
        calls = [(g, (t,), ang() if g in ("RZ", "RY") else us[t] if g == "U2" else ())
                 for g in ("X", "H", "RZ", "RY", "U2") for t in range(n)]
        return calls + [(g, (a, b), ()) for g in ("CNOT", "CZ", "SWAP") for a in range(n) for b in range(n) if a != b]
    calls = []
    targets = sorted({0, 1, n // 3, n // 2, n - 2, n - 1})
    us = haar(4, len(targets), seed + 1)
    for t, u in zip(targets, us):
        c = n - 4 if t != n - 4 else 0
        calls += [("H", (t,), ()), ("RZ", (t,), ang()), ("CNOT", (c, t), ()), ("U4", (t, (t + 1) % n), u)]
    return calls


def batch_shapes(case):
    r = random.Random(7)
    return [(r.randint(case["n_min"], case["n_max"]), r.randint(4, 12)) for _ in range(case["count"])]


def angles(case, seed):
    return np.random.default_rng(seed).uniform(0, 2 * math.pi, 2 * case["n"] * case["layers"])


def batch_angles(case, seed):
    r = np.random.default_rng(seed)
    return [r.uniform(0, 2 * math.pi, 2 * n * l) for n, l in batch_shapes(case)]


def random_state(n, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(1 << n, dtype=TORCH[dtype], device="cuda", generator=g)
    return x.div_(torch.linalg.vector_norm(x))


# ---------------------------------------------------------------------------
# the measured call
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind, dt = case["kind"], case["dtype"]
    if kind == "batch":
        shapes, terms = batch_shapes(case), {n: tfim(n) for n in range(case["n_min"], case["n_max"] + 1)}
        circuits = [Circuit(n, ansatz_ops(n, l), p) for (n, l), p in zip(shapes, batch_angles(case, seed))]
        return {"kind": kind, "dtype": dt, "items": L.BatchItems(circuits, [terms[c.n_qubits] for c in circuits])}
    n = case["n"]
    s = {"kind": kind, "params": None}
    if kind in ("ansatz", "gradient"):
        ops, s["params"] = ansatz_ops(n, case["layers"]), angles(case, seed)
        s["sv"] = L.StateVector(n, dt)
    else:
        s["sv"] = L.StateVector(n, dt, tensor=random_state(n, dt, seed))
        if kind == "gates":
            s["calls"] = gate_calls(case, seed)
            return s
        if kind == "qft":
            _, ops, s["params"] = qft_circuit(n)
        elif kind == "universal":
            _, ops, s["params"] = universal_circuit(n)
        elif kind == "windows":
            ops = window_ops(case, seed)
    # a program that repeats a circuit marshals it once and has its kernels compiled ahead of its loop
    if kind in ("expval", "gradient"):
        s["terms"] = L.PauliArray(tfim(n))
        if n >= 20:
            L.lqs_jit_precompile_expval(n, dt, s["terms"])
    if kind != "expval":
        s["ops"] = L.OpArray(ops)
        if n >= 20:
            L.lqs_jit_precompile(n, dt, s["ops"], s["params"])
    if kind == "gradient" and n >= 20:
        L.lqs_jit_precompile_expval(n, dt, s["terms"], lambda_=True)
        L.lqs_jit_precompile_adjoint(n, dt, s["ops"], s["params"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        energies, grads = s["items"].run(s["dtype"])
        return {"energies": energies, "grads": np.concatenate(grads)}
    sv = s["sv"]
    if kind == "gates":
        for gate, wires, params in s["calls"]:
            sv.apply_gate(gate, wires, params)
        return {"state": sv.tensor}
    if kind == "expval":
        energy, words = sv.expval(s["terms"])
        return {"energy": np.float64(energy), "words": words}
    if kind in ("ansatz", "gradient"):
        sv.set_basis(0)
    L.lqs_apply_fused(sv.h, s["ops"], s["params"])
    if kind != "gradient":
        return {"state": sv.tensor}
    energy, words = sv.expval(s["terms"])
    grads, again = L.lqs_adjoint_grad(sv.h, s["ops"], s["params"], s["terms"])
    return {"energy": np.float64(energy), "energy_of_gradient": np.float64(again), "words": words, "grads": grads,
            "state": sv.tensor}


def work(case):
    """Bytes: the state read and written once (the ansatz and the gradients start from |0..0>: no state is read).
    Flops per amplitude: 6 per real 2x2 or complex factor, 4 per Hadamard, 14 and 30 per dense one- and two-qubit
    gate; diagonal gates that follow one another count as one factor."""
    def train(n, l):  # forward, un-applying two states, the generators' sums, lambda and the energy
        return 2.0 ** n * (3 * l * (6 * n + 6) + l * (8 * n + 3 + n) + 4 * n + 6 * n)

    kind, b = case["kind"], AMP[case["dtype"]]
    if kind == "batch":
        shapes = batch_shapes(case)
        return {"bytes": sum(2 * 8.0 * 2 * n * l for n, l in shapes), "flops": sum(train(n, l) for n, l in shapes)}
    n = case["n"]
    N = 2.0 ** n
    if kind == "gates":
        per = {"X": (1, 0), "H": (1, 4), "RZ": (1, 6), "RY": (1, 6), "U2": (1, 14), "CNOT": (.5, 0), "CZ": (.25, 1),
               "SWAP": (.5, 0), "U4": (1, 30)}
        calls = [per[g] for g, _, _ in gate_calls(case, 0)]
        return {"bytes": sum(2 * b * N * f for f, _ in calls), "flops": sum(N * x for _, x in calls)}
    if kind == "ansatz":
        return {"bytes": b * N, "flops": N * case["layers"] * (6 * n + 6)}
    if kind == "qft":
        return {"bytes": 2 * b * N, "flops": N * (4 * n + 6 * (n - 1))}
    if kind == "universal":
        return {"bytes": 2 * b * N, "flops": N * 6 * (n + 1)}
    if kind == "windows":
        return {"bytes": 2 * b * N, "flops": N * 30 * case["windows"] * case["gates"]}
    if kind == "expval":
        return {"bytes": b * N, "flops": N * (3 + n - 1 + 4 * n)}
    return {"bytes": b * N, "flops": train(n, case["layers"])}


# ---------------------------------------------------------------------------
# the same in plain torch, complex128
# ---------------------------------------------------------------------------

def _one(v, q, u):
    """A 2x2 matrix on qubit q of each row of v."""
    x = v.view(v.shape[0], -1, 2, 1 << q)
    a, b = x[:, :, 0].clone(), x[:, :, 1]
    x[:, :, 0].mul_(complex(u[0][0])).add_(b, alpha=complex(u[0][1]))
    b.mul_(complex(u[1][1])).add_(a, alpha=complex(u[1][0]))


def _two(v, wires, u):
    """A 4x4 matrix on (most, least significant) wires of each row of v."""
    hi, lo = max(wires), min(wires)
    x = v.view(v.shape[0], -1, 2, 1 << (hi - lo - 1), 2, 1 << lo)
    part = [x[:, :, (j >> 1, j & 1)[wires[0] != hi], :, (j >> 1, j & 1)[wires[0] == hi]] for j in range(4)]
    old = [p.clone() for p in part]
    for j, p in enumerate(part):
        p.mul_(complex(u[j][j]))
        for k in range(4):
            if k != j and u[j][k] != 0:
                p.add_(old[k], alpha=complex(u[j][k]))


def _phase(v, q, f0, f1):
    x = v.view(v.shape[0], -1, 2, 1 << q)
    if f0 != 1:
        x[:, :, 0].mul_(f0)
    x[:, :, 1].mul_(f1)


def _ry(t):
    return [[math.cos(t / 2), -math.sin(t / 2)], [math.sin(t / 2), math.cos(t / 2)]]


def _ladder(v, n, inverse=False):
    """CNOT(0,1), CNOT(1,2), ...: bit i becomes the parity of bits 0..i."""
    y = torch.arange(1 << n, device=v.device)
    if inverse:
        s = 1
        while s < n:
            y ^= (y << s) & ((1 << n) - 1)
            s *= 2
    else:
        y ^= (y << 1) & ((1 << n) - 1)
    return torch.stack([r[y] for r in v]) if v.shape[0] > 1 else v[0][y].unsqueeze(0)


def _zero(n):
    v = torch.zeros(1, 1 << n, dtype=torch.complex128, device="cuda")
    v[0, 0] = 1
    return v


def _forward(n, layers, p):
    v = _zero(n)
    for l in range(layers):
        for q in range(n):
            _one(v, q, _ry(p[2 * n * l + q]))
        for q in range(n):
            t = p[2 * n * l + n + q]
            _phase(v, q, complex(math.cos(t / 2), -math.sin(t / 2)), complex(math.cos(t / 2), math.sin(t / 2)))
        v = _ladder(v, n)
    return v


def _words(v, n):
    """<Z_i Z_i+1> for each i, then <X_i> for each i, of one row."""
    w = v.real.square() + v.imag.square()
    out = []
    for i in range(n - 1):
        x = w.view(-1, 2, 2, 1 << i).sum(dim=(0, 3))
        out.append(x[0, 0] + x[1, 1] - x[0, 1] - x[1, 0])
    for i in range(n):
        x = v.view(-1, 2, 1 << i)
        out.append(2 * (x[:, 0].real * x[:, 1].real + x[:, 0].imag * x[:, 1].imag).sum())
    return torch.stack(out)


def _gradient(n, layers, p):
    """Words of the output state and the adjoint gradient of the TFIM energy."""
    v = _forward(n, layers, p)
    words = _words(v[0], n)
    lam = torch.zeros_like(v[0])
    j = torch.arange(1 << n, device="cuda")
    zz = torch.zeros(1 << n, dtype=torch.float64, device="cuda")
    for i in range(n - 1):
        zz += 1 - 2 * (((j >> i) ^ (j >> (i + 1))) & 1)
    lam += zz * v[0]
    for i in range(n):
        lam.view(-1, 2, 1 << i).add_(v[0].view(-1, 2, 1 << i).flip(1), alpha=0.5)
    del zz, j
    s = torch.stack([v[0], lam])
    g = [None] * len(p)
    for l in range(layers - 1, -1, -1):
        s = _ladder(s, n, inverse=True)
        w = s[1].real * s[0].imag - s[1].imag * s[0].real  # Im conj(lambda) psi
        for q in range(n):
            x = w.view(-1, 2, 1 << q).sum(dim=(0, 2))
            g[2 * n * l + n + q] = x[0] - x[1]
            t = p[2 * n * l + n + q]
            _phase(s, q, complex(math.cos(t / 2), math.sin(t / 2)), complex(math.cos(t / 2), -math.sin(t / 2)))
        for q in range(n - 1, -1, -1):
            x = s.view(2, -1, 2, 1 << q)
            a, b = x[:, :, 0], x[:, :, 1]  # Im <lambda|Y|psi> = sum Re(conj(l1) p0 - conj(l0) p1)
            g[2 * n * l + q] = (b[1].real * a[0].real + b[1].imag * a[0].imag - a[1].real * b[0].real
                                - a[1].imag * b[0].imag).sum()
            _one(s, q, _ry(-p[2 * n * l + q]))
    coeff = torch.tensor([1.0] * (n - 1) + [0.5] * n, dtype=torch.float64, device="cuda")
    return words, (words * coeff).sum(), torch.stack(g)


def exact(case, seed):
    kind, dt = case["kind"], case["dtype"]
    if kind == "batch":
        got = [_gradient(n, l, list(p)) for (n, l), p in zip(batch_shapes(case), batch_angles(case, seed))]
        return {"energies": torch.stack([e for _, e, _ in got]), "grads": torch.cat([g for _, _, g in got])}
    n = case["n"]
    if kind == "ansatz":
        return {"state": _forward(n, case["layers"], list(angles(case, seed)))[0]}
    if kind == "gradient":
        words, e, g = _gradient(n, case["layers"], list(angles(case, seed)))
        return {"energy": e, "energy_of_gradient": e, "words": words, "grads": g, "state": _zero(n)[0]}
    v = random_state(n, dt, seed).to(torch.complex128).unsqueeze(0)
    if kind == "expval":
        words = _words(v[0], n)
        coeff = torch.tensor([1.0] * (n - 1) + [0.5] * n, dtype=torch.float64, device="cuda")
        return {"energy": (words * coeff).sum(), "words": words}
    if kind == "qft":
        return {"state": torch.fft.ifft(v[0], norm="ortho")}
    if kind == "universal":
        for layer in range(n + 1):
            for q in range(n):
                t = universal_angle(layer, q, n)
                _phase(v, q, 1, complex(math.cos(t), math.sin(t)))
            if layer < n:
                v = _ladder(v, n)
        return {"state": v[0]}
    if kind == "windows":
        for w, u in zip(window_wires(case), haar(4, len(window_wires(case)), seed)):
            _two(v, w, u)
        return {"state": v[0]}
    h = 1 / math.sqrt(2)
    for gate, wires, p in gate_calls(case, seed):
        if len(wires) == 2:
            m = {"CNOT": [0, 1, 3, 2], "SWAP": [0, 2, 1, 3]}.get(gate)
            _two(v, wires, np.eye(4)[m] if m else np.diag([1, 1, 1, -1]) if gate == "CZ" else p)
        elif gate == "RZ":
            _phase(v, wires[0], complex(math.cos(p[0] / 2), -math.sin(p[0] / 2)),
                   complex(math.cos(p[0] / 2), math.sin(p[0] / 2)))
        else:
            _one(v, wires[0], {"X": [[0, 1], [1, 0]], "H": [[h, h], [h, -h]]}.get(gate) or
                 (_ry(p[0]) if gate == "RY" else p))
    return {"state": v[0]}
