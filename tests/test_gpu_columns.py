"""The FP32 circuit unitary as a batch of columns: every thread count the launch
takes (1 to 16 warps, two groups per thread at n = 14), blocks that are not
whole transpose tiles, SWAPs, leading and trailing X, custom gates, and a
circuit changed between calls.  Tolerance 1e-5, the FP32 form's."""
import numpy as np
import pytest

from oracle import fsv_route
from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W
from test_host_program import with_customs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def columns(c, n, col0, ncols, ldu):
    U = torch.full((1 << n, ldu), float("nan"), dtype=torch.complex64, device="cuda")
    B.tqs_circuit_unitary_cols(c, B.PREC_FP32_SIMT, col0, ncols, U, ldu=ldu)
    got = U.cpu().numpy()
    assert np.all(np.isnan(got[:, ncols:]))
    return got[:, :ncols]


@pytest.mark.parametrize("n", [2, 4, 6, 9, 10, 11, 13, 14])
def test_columns_match_oracle(n):
    ops = [("x", (0,), ())] + list(W.random_small(n, 6 * n, (95, n))) + [("swap", (0, n - 1), ()), ("x", (n - 1,), ())]
    N = 1 << n
    col0, ncols = (1, N - 2) if n < 7 else (N - 128, 128)
    c = B.circuit_from_ops(n, ops)
    try:
        got = columns(c, n, col0, ncols, ncols + 3)
        pick = sorted({0, 1, ncols // 2, ncols - 1})
        want = fsv_route.unitary_columns(n, ops, [col0 + p for p in pick])
        assert np.max(np.abs(got[:, pick] - want)) <= 1e-5
        B.tqs_add_gate(c, "h", (0,))  # the program that the handle holds is built again
        got = columns(c, n, col0, ncols, ncols)
        want = fsv_route.unitary_columns(n, ops + [("h", (0,), ())], [col0 + p for p in pick])
        assert np.max(np.abs(got[:, pick] - want)) <= 1e-5
    finally:
        B.tqs_circuit_destroy(c)


@pytest.mark.parametrize("n", [3, 7])
def test_columns_with_custom_gates(n):
    ops, _ = with_customs(n, 96 + n)
    c = B.circuit_from_ops(n, ops)
    try:
        got = columns(c, n, 0, 1 << n, 1 << n)
        want = fsv_route.unitary_columns(n, ops, list(range(1 << n)))
        assert np.max(np.abs(got - want)) <= 1e-5
    finally:
        B.tqs_circuit_destroy(c)
