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
