"""Fusion planner checks (host logic, no GPU).

The plan may reorder gates only across gates on disjoint wires.  Executing the
ops segment by segment (original relative order inside a segment) through the
CPU oracle must therefore reproduce the in-order result; and every segment's
tile must hold the low qubits and every non-diagonal target of its gates.
"""
import ctypes
import math
import os
import time

import numpy as np
import pytest

import oracle
import paper_2508_13615_gb300 as L
import workloads as W

DIAG = {"Z", "S", "T", "RZ", "PhaseShift", "CZ", "ControlledPhaseShift"}


def planned_order(c, cfg=None, dtype="c128"):
    nseg, masks, seg_of = L.lqs_plan_fused(c.n_qubits, dtype, c.ops, cfg)
    assert all(0 <= s < nseg for s in seg_of)
    order = sorted(range(len(c.ops)), key=lambda i: (seg_of[i], i))
    return nseg, masks, seg_of, order


def run_in_order(c, order, psi0):
    cc = W.Circuit(c.n_qubits, [c.ops[i] for i in order], c.params)
    return oracle.run_circuit(cc, psi0)


@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("cfg", [None, {"tile_qubits": 5, "low_qubits": 2}, {"tile_qubits": 4, "low_qubits": 1},
                                 {"tile_qubits": 6, "low_qubits": 3, "max_ops": 5}])
def test_planned_order_reproduces_circuit(seed, cfg):
    n = 9
    # gates that run as one kernel op (DoubleExcitation runs as nine, which the
    # planner may interleave with other gates, so it has no single segment)
    names = [g for g, _, _ in W.GATES if g != "DoubleExcitation"]
    c = W.random_circuit(n, 80, seed=100 + seed, names=names)
    psi0 = W.gaussian_state(n, seed)
    nseg, masks, seg_of, order = planned_order(c, cfg)
    np.testing.assert_allclose(run_in_order(c, order, psi0), oracle.run_circuit(c, psi0), atol=1e-12)


def test_segment_tiles_hold_targets_and_low_qubits():
    n = 20
    c = W.random_circuit(n, 300, seed=5)
    cfg = {"tile_qubits": 8, "low_qubits": 3}
    nseg, masks, seg_of, _ = planned_order(c, cfg)
    for m in masks:
        assert bin(m).count("1") == 8 and (m & 0b111) == 0b111
    for i, op in enumerate(c.ops):
        if op.name in DIAG:
            continue
        m = masks[seg_of[i]]
        targets = op.wires[-1:] if op.name not in ("SWAP", "U4") else op.wires
        if op.name in ("U2", "Rot", "RX", "RY", "H", "X", "Y", "CNOT", "CRY", "Toffoli"):
            targets = op.wires[-1:]
        for t in targets:
            assert (m >> t) & 1, (op.name, op.wires, hex(m))


def test_fusion_cuts_passes_at_least_fourfold():
    for c in (W.ansatz(30, 10, 3), W.qft(30), W.ansatz(24, 8, 6)):
        for dt in ("c128", "c64"):
            nseg = L.lqs_plan_fused(c.n_qubits, dt, c.ops)[0]
            assert len(c.ops) / nseg >= 4, (len(c.ops), nseg)


def test_small_state_is_one_tile():
    c = W.ansatz(6, 3, 1)
    nseg, masks, _, _ = planned_order(c)
    assert nseg == 1 and masks[0] == (1 << 6) - 1


@pytest.mark.parametrize("name,n,dtype", [("ansatz", 15, "c128"), ("ansatz", 16, "c64"), ("qft", 15, "c128"),
                                          ("universal", 15, "c128"), ("random", 15, "c128"), ("random", 16, "c64")])
def test_searched_plans_reproduce_the_circuit(name, n, dtype):
    """Plans of compiled segments look for fuller tiles and let ops pass each other on wires that both leave in the
    Z basis: the planned order must still give the in-order state, every non-diagonal target must sit in its
    segment's tile, and no searched plan may need more passes than program order does."""
    if name == "random":
        names = [g for g, _, _ in W.GATES if g != "DoubleExcitation"]
        c = W.random_circuit(n, 120, seed=7, names=names)
    else:
        c = W.ansatz(n, 4, 3) if name == "ansatz" else getattr(W, name)(n)
    psi0 = W.gaussian_state(n, 5)
    old = L.lqs_jit_info()["mode"]
    try:
        L.lqs_set_jit(L.LQS_JIT_ON)
        nseg, masks, seg_of, order = planned_order(c, None, dtype)
        L.lqs_set_jit(L.LQS_JIT_OFF)  # no compiled kernels, no dense cap: program order
        plain = planned_order(c, {"max_ops": 16}, dtype)[0]
    finally:
        L.lqs_set_jit(old)
    np.testing.assert_allclose(run_in_order(c, order, psi0), oracle.run_circuit(c, psi0), atol=1e-12)
    for i, op in enumerate(c.ops):
        if op.name not in DIAG and op.name not in ("U2", "U4"):
            targets = op.wires[-2:] if op.name in ("SWAP", "CSWAP") else op.wires[-1:]
            assert all((masks[seg_of[i]] >> t) & 1 for t in targets), (op.name, op.wires)
    assert nseg <= plain


def test_four_two_qubit_gates_share_a_compiled_segment():
    """The cap on a compiled complex128 segment's dense work leaves room for four two-qubit matrices: eight of them in
    one tile take two passes."""
    n = 14
    c = W.Circuit(n)
    for i in range(8):
        c.add("U4", (i % 5, 5 + i % 4), matrix=W.haar_unitary(4, i))
    old = L.lqs_jit_info()["mode"]
    try:
        L.lqs_set_jit(L.LQS_JIT_ON)
        assert L.lqs_plan_fused(n, "c128", c.ops, None)[0] == 2
    finally:
        L.lqs_set_jit(old)


def program_order_passes(c, k, b, cap, w2):
    """Passes of the plain greedy plan: a segment takes every op, in program order, that shares no wire with an op it
    has left behind and whose non-diagonal targets fit the tile, up to 128 ops and the cap on dense work."""
    dense = {"H": 1, "RX": 1, "RY": 1, "Rot": 1, "U2": 1, "CRY": 1, "U4": w2}
    left, passes = list(range(len(c.ops))), 0
    while left:
        tile, blocked, work, taken, rest = set(range(b)), set(), 0, 0, []
        for i in left:
            op = c.ops[i]
            t = set() if op.name in DIAG else set(op.wires[-2:] if op.name in ("SWAP", "CSWAP", "U4") else op.wires[-1:])
            w = dense.get(op.name, 0)
            if not (blocked & set(op.wires)) and len(tile | t) <= k and taken < 128 and (work + w <= cap or not taken):
                tile, work, taken = tile | t, work + w, taken + 1
            else:
                blocked |= set(op.wires)
                rest.append(i)
        assert len(rest) < len(left)
        left, passes = rest, passes + 1
    return passes


@pytest.mark.parametrize("name", ["ansatz", "qft", "universal", "random"])
def test_searched_plans_against_program_order(name):
    """Double-float plans of compiled segments never take more passes than program order under the same cap on dense
    work, and fewer where layers overlap (ansatz, universal circuit).  The float64 policy and complex64 keep program
    order: exactly its number of passes."""
    n = 18
    if name == "random":
        c = W.random_circuit(n, 120, seed=7, names=[g for g, _, _ in W.GATES if g != "DoubleExcitation"])
    else:
        c = W.ansatz(n, 6, 3) if name == "ansatz" else getattr(W, name)(n)
    old = L.lqs_jit_info()["mode"]
    try:
        L.lqs_set_jit(L.LQS_JIT_ON)
        passes = {a: L.lqs_plan_fused(n, "c128", c.ops, {"arith": a})[0] for a in (L.LQS_ARITH_DF, L.LQS_ARITH_F64)}
        c64 = L.lqs_plan_fused(n, "c64", c.ops, None)[0]
    finally:
        L.lqs_set_jit(old)
    plain = program_order_passes(c, 12, 4, 12, 3)
    assert passes[L.LQS_ARITH_DF] < plain if name in ("ansatz", "universal") else passes[L.LQS_ARITH_DF] <= plain
    assert passes[L.LQS_ARITH_F64] == program_order_passes(c, 12, 4, 24, 3)
    assert c64 == program_order_passes(c, 13, 5, 64, 4)


def test_planning_time_is_proportional_to_the_circuit():
    """Phase-estimation shape: one wire is never a target, so it never blocks.  Planning eight times the ops may take
    twice its share of the time, far from the 64 of a search that scans the whole circuit for every segment."""
    n = 30

    def seconds(m, seed):
        r = W.splitmix64(seed, 0, m)
        c = W.Circuit(n)
        c.params = np.array([0.3])
        for i in range(m):
            q = 1 + int(r[i] % np.uint64(n - 1))
            c.ops.append([W.Op("RY", (q,), 0), W.Op("ControlledPhaseShift", (0, q), 0),
                          W.Op("CNOT", (q, 1 + q % (n - 1)))][i % 3])
        ops = L.OpArray(c.ops)
        t0 = time.process_time()
        L.lqs_plan_fused(n, "c128", ops, None)
        return time.process_time() - t0

    old = L.lqs_jit_info()["mode"]
    try:
        L.lqs_set_jit(L.LQS_JIT_ON)
        small = min(seconds(4000, s) for s in (1, 2, 3))
        assert seconds(32000, 4) <= 16 * small
    finally:
        L.lqs_set_jit(old)


def test_kept_plans_are_bounded_in_bytes():
    """Sixty plans of 100000 ops (2.8 MB each with their keys) leave no more than the store's 32 MiB behind, and as much
    again for what the allocator keeps."""
    def resident():
        ctypes.CDLL(None).malloc_trim(0)  # freed blocks between live ones
        with open("/proc/self/statm") as f:
            return int(f.read().split()[1]) * os.sysconf("SC_PAGE_SIZE")

    c = W.Circuit(13)
    c.ops = [W.Op("X", (i % 12,)) for i in range(100000)]
    ops = L.OpArray(c.ops)
    old = L.lqs_jit_info()["mode"]
    try:
        L.lqs_set_jit(L.LQS_JIT_ON)
        L.lqs_plan_fused(13, "c128", ops, {"max_ops": 60})
        before = resident()
        for max_ops in range(61, 121):
            L.lqs_plan_fused(13, "c128", ops, {"max_ops": max_ops})
        assert resident() - before <= 2 * (32 << 20)
    finally:
        L.lqs_set_jit(old)
