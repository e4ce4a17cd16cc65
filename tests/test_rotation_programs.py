"""Programs with rotations: general single-qubit gates split into a phase and a
rotation, their outer factors (phases, X, X-axis factors) carried through the
circuit (prepare_gates).  Circuits that reach every move of a pending factor
(controls, targets, controlled phases under an X, SWAP, instructions' and
custom gates' barriers, the circuit's end) and the angles where a split is
degenerate, on the CPU replay of the compiled program and on the GPU.

Tolerances: the replay computes in FP64 with the program's FP32 coefficients
(2e-6, as for every program); the kernels keep FP32 amplitudes (1e-5).
"""
import math

import numpy as np
import pytest

import test_host_program as hp
from oracle import fsv_route
from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W

ANGLES = [0.0, 1e-9, 1e-5, math.pi / 2, math.pi - 1e-9, math.pi, math.pi + 1e-6, 2 * math.pi, 3.0]
ONE = ["h", "x", "y", "z", "s", "t", "r", "rx", "ry", "rz", "u3"]
TWO = ["cx", "cz", "cp", "cu", "swap"]


def carried(n, count, seed):
    """A random circuit whose angles are half degenerate and whose two-qubit
    gates meet every pending factor."""
    g = W.rng(71, n, seed)
    ops = []
    for _ in range(count):
        two = n > 1 and g.random() < 0.5
        name = (TWO if two else ONE)[int(g.integers(0, 5 if two else len(ONE)))]
        qs = tuple(int(q) for q in g.permutation(n)[: 2 if two else 1])
        if name == "cu":
            ps = W.random_small(2, 1, (72, n, seed, len(ops)), names=("cu",))[0][2]
        else:
            ps = tuple(float(ANGLES[int(g.integers(0, len(ANGLES)))] if g.random() < 0.5 else g.uniform(0, 7))
                       for _ in range(W.N_PARAMS[name]))
        ops.append((name, qs, ps))
    return ops


def two_angles(name, a, b):
    """A degenerate gate on each side of a CNOT target, of a control and of a
    controlled phase, an X before each."""
    p = (a, b, 0.7) if name == "u3" else (a,)
    q = (b, 0.3, a) if name == "u3" else (b,)
    ops = []
    for mid in (("cx", (0, 1), ()), ("cx", (1, 0), ()), ("cp", (1, 2), (0.9,)), ("cz", (2, 1), ())):
        ops += [(name, (1,), p), ("x", (1,), ()), mid, (name, (1,), q), ("x", (2,), ()), ("h", (2,), ())]
    return ops


CASES = [(n, carried(n, 12 * n, s)) for n in (1, 2, 3, 5, 8, 11) for s in range(4)]
CASES += [(3, two_angles(name, a, b)) for name in ("rx", "ry", "rz", "u3") for a, b in
          [(0.0, 2.0), (math.pi, 1.0), (math.pi - 1e-9, math.pi), (1e-9, math.pi / 2), (3.148, 2.705)]]
IDS = [f"n{n}-{i}" for i, (n, _) in enumerate(CASES)]


@pytest.mark.parametrize("n,ops", CASES, ids=IDS)
def test_replay_matches_oracle(n, ops):
    got = hp.replay(n, *hp.compiled(n, ops))
    assert np.max(np.abs(got - fsv_route.simulate(n, ops))) < 2e-6


def test_deep_circuit_keeps_its_scale():
    """Unscaled rotations over many passes: the factor held back is applied in
    time (a 3-qubit circuit of 3000 gates)."""
    ops = W.random_layered(3, 700, (73, 1))
    got = hp.replay(3, *hp.compiled(3, ops))
    assert np.max(np.abs(got - fsv_route.simulate(3, ops))) < 2e-5  # 2100 roundings of FP32 angles, at most 1.5e-8 each


@pytest.mark.gpu
@pytest.mark.parametrize("n", [1, 4, 8, 11, 12, 14, 15])
def test_gpu_fused_and_tiled(n):
    import torch
    for s in range(2):
        ops = carried(n, 8 * n, 10 + s)
        want = fsv_route.simulate(n, ops)
        c = B.circuit_from_ops(n, ops)
        try:
            out = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
            B.tqs_simulate(c, out)
            st = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
            st[0] = 1.0
            B.tqs_simulate_fsv(c, st)
            init = torch.zeros_like(out)
            init[0] = 1.0
            again = torch.empty_like(out)
            B.tqs_simulate(c, again, init=init)
            for v in (out, st, again):
                assert np.max(np.abs(v.cpu().numpy() - want)) <= 1e-5
        finally:
            B.tqs_circuit_destroy(c)


@pytest.mark.gpu
def test_gpu_tiled_per_gate_form():
    """One gate per pass: every rotation's outer factors stay in its pass."""
    import torch
    n, ops = 14, carried(14, 80, 3)
    c = B.circuit_from_ops(n, ops)
    try:
        B.tqs_set_option(B.OPT_FSV_MAX_GATES, 0, 1)
        st = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
        st[0] = 1.0
        B.tqs_simulate_fsv(c, st)
        assert np.max(np.abs(st.cpu().numpy() - fsv_route.simulate(n, ops))) <= 1e-5
    finally:
        B.tqs_set_option(B.OPT_FSV_MAX_GATES, 0, 0)
        B.tqs_circuit_destroy(c)
