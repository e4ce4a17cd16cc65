"""How exactly a program holds its rotations: the compiled program's
coefficients, on the CPU replay (FP64 arithmetic, so their error alone),
against the FP64 oracle, and the same circuits on the GPU.
"""
import math

import numpy as np
import pytest

import test_host_program as hp
from oracle import fsv_route
from paper_2305_14398_gb300 import binding as B

TINY = [1e-9, 1e-10, 1e-11, 1e-12, 1e-13, 3e-14, 1e-14, 3e-15]
TINY += [math.pi + a for a in TINY] + [-a for a in TINY[1:6]] + [2000 * math.pi, 2001 * math.pi]


def tiny_turn(name, a):
    """X-rotations times a turn by the angle a about another axis before a
    CNOT's target: what an X-axis factor leaves has a tiny real entry."""
    ops = []
    for x in (0.4, 1.3, math.pi - 0.2, 2.9):
        ops += [("rz", (1,), (0.8 + x,)), ("rx", (1,), (x,)), (name, (1,), (a,)), ("cx", (0, 1), ()),
                ("h", (0,), ()), (name, (0,), (a,)), ("rx", (0,), (x,)), ("cx", (1, 0), ())]
    return ops


@pytest.mark.parametrize("a", TINY)
@pytest.mark.parametrize("name", ["ry", "rz"])
def test_tiny_turns_after_x_rotations(name, a):
    # one FP32 rounding of the start's factor and of each of 8 angles
    ops = tiny_turn(name, a)
    got = hp.replay(2, *hp.compiled(2, ops))
    assert np.max(np.abs(got - fsv_route.simulate(2, ops))) < 2e-7


REPEATED = [0.01, 0.7, 0.9274, 1.0, 1.5707963, 2.0, 3.0]


def repeated(n, count, name, theta):
    """The same turn on every qubit between layers of CZ, `count` times."""
    layer = [(name, (q,), (theta, 0.4, 1.1) if name == "u3" else (theta,)) for q in range(n)]
    layer += [("cz", (q, q + 1), ()) for q in range(n - 1)]
    return layer * count


@pytest.mark.parametrize("theta", REPEATED)
@pytest.mark.parametrize("name", ["ry", "rx", "u3"])
def test_repeated_angles_do_not_drift(name, theta):
    # an angle is held to 2^-37: 2000 turns of two qubits are off by 1.5e-8 at
    # most, beside the start's factor, one FP32 rounding (6e-8)
    ops = repeated(2, 1000, name, theta)
    got = hp.replay(2, *hp.compiled(2, ops))
    assert np.max(np.abs(got - fsv_route.simulate(2, ops))) < 2e-7


def with_low_parts(prog):
    """The program with the hi + lo phases that follow rotations (field c of an
    uncontrolled local diagonal op) as FP64, which the replay reads as hi alone."""
    ops = prog[1]
    wide = np.zeros(len(ops), dtype=[(k, (np.complex128, (4,))) if k == "m" else (k,) + (
        ops.dtype[k].subdtype if ops.dtype[k].subdtype else (ops.dtype[k],)) for k in ops.dtype.names])
    for k in ops.dtype.names:
        wide[k] = ops[k]
    hl = (ops["code"] >= 40) & (ops["code"] < 44) & (ops["c"] == 1)
    wide["m"][hl, 1] += ops["lo"][hl, 0]
    wide["m"][hl, 2] = wide["m"][hl, 1]
    return (prog[0], wide) + tuple(prog[2:])


@pytest.mark.parametrize("theta", [0.7, 2.0, math.pi, math.pi - 1e-15])
def test_repeated_phases_do_not_drift(theta):
    # phases before controls, targets and half turns: as for the angles
    ops = [("u3", (q,), (theta, 0.3, 0.9)) for q in range(3)]
    ops = (ops + [("cx", (0, 1), ()), ("ry", (0,), (0.5,)), ("cx", (1, 2), ()), ("rz", (2,), (0.4,))]) * 700
    got = hp.replay(3, *with_low_parts(hp.compiled(3, ops)))
    assert np.max(np.abs(got - fsv_route.simulate(3, ops))) < 2e-7


@pytest.mark.gpu
@pytest.mark.parametrize("theta", [0.7, 0.9274, 1.0, 2.0])
def test_gpu_repeated_angles(theta):
    """3000 layers on 6 qubits: an amplitude, about 1/8, is rounded 36000 times,
    each by 0.29 * 2^-23 of its size on average: 190 * 3.5e-8 / 8 = 8e-7
    expected, five times that allowed (a drift of 2.4e-8 a turn gives 1.9e-5).
    A CTA, a tile (all gates that fit, and 64 at a time), a warp (in a batch too
    large for a CTA each)."""
    import torch
    n = 6
    ops = repeated(n, 3000, "ry", theta)
    want = fsv_route.simulate(n, ops)
    c = B.circuit_from_ops(n, ops)
    small = B.circuit_from_ops(1, [("h", (0,), ())])
    b = B.tqs_batch_create([c] + [small] * 1300)
    try:
        out = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
        B.tqs_simulate(c, out)
        tile = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
        tile[0] = 1.0
        B.tqs_simulate_fsv(c, tile)
        bounded = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
        bounded[0] = 1.0
        B.tqs_set_option(B.OPT_FSV_MAX_GATES, 0, 64)
        B.tqs_simulate_fsv(c, bounded)
        st = torch.empty((1 << n) + 2 * 1300, dtype=torch.complex64, device="cuda")
        B.tqs_batch_run(b, st)
        for v in (out, tile, bounded, st[:1 << n]):
            assert np.max(np.abs(v.cpu().numpy() - want)) < 4e-6
    finally:
        B.tqs_set_option(B.OPT_FSV_MAX_GATES, 0, 0)
        B.tqs_batch_destroy(b)
        B.tqs_circuit_destroy(small)
        B.tqs_circuit_destroy(c)


@pytest.mark.gpu
@pytest.mark.parametrize("name,theta,tol", [("ry", 0.9274, 4e-6), ("ry", 2.0, 4e-6), ("u3", 0.9274, 6e-6), ("u3", 2.0, 6e-6)])
def test_gpu_repeated_steps(name, theta, tol):
    """One layer as a circuit of its own, applied 3000 times to what it returned:
    the same bound, though each of its angles occurs few times.  A U3's two phases
    round an amplitude about three times more per turn: 90000 in all."""
    import torch
    n = 6
    want = fsv_route.simulate(n, repeated(n, 3000, name, theta))
    c = B.circuit_from_ops(n, repeated(n, 1, name, theta))
    try:
        st = [torch.zeros(1 << n, dtype=torch.complex64, device="cuda") for _ in range(2)]
        tile = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
        st[0][0] = tile[0] = 1.0
        for k in range(3000):
            B.tqs_simulate(c, st[1 - k % 2], init=st[k % 2])
            B.tqs_simulate_fsv(c, tile)
        for v in (st[0], tile):
            assert np.max(np.abs(v.cpu().numpy() - want)) < tol
    finally:
        B.tqs_circuit_destroy(c)
