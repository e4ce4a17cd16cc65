"""Step matrices of 10 and 11 qubits on either side of the number of factors from
which rows are expanded: two-qubit and custom factors among them, idle qubits.
Sampled columns against the oracle's, 1e-6 (products of at most 11 FP32 entries)."""
import numpy as np
import pytest

from oracle import fsv_route
from oracle import gates as G
from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W
from test_host_program import rand_unitary

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,factors", [(10, 8), (10, 9), (11, 4), (11, 5), (11, 9)])
def test_columns_by_number_of_factors(n, factors):
    t = n - 1
    ops = [("cu", (t, 0), W.random_small(2, 1, (96, n), names=("cu",))[0][2])]
    if n == 11:
        ops.append(("unitary", (t - 1, 1, 5), G.custom_params(rand_unitary(3, n))))
    free = [q for q in range(n) if q not in {t, 0} | ({t - 1, 1, 5} if n == 11 else set())]
    if len(ops) + len(free) < factors:  # nine factors of 11 qubits: no custom one
        ops, free = ops[:1], [q for q in range(n) if q not in (t, 0)]
    ops += [("u3", (q,), (0.3 + q, 0.2, 0.1)) for q in free[:factors - len(ops)]]
    assert len(ops) == factors
    cols = sorted({0, 1, (1 << n) - 1, 1 << (n - 3), 5 * 41 + 7, (1 << n) - 6})
    c = B.circuit_from_ops(n, ops)
    try:
        S = torch.full((1 << n, 1 << n), float("nan"), dtype=torch.complex64, device="cuda")
        B.tqs_materialize_step(c, 0, S)
        assert not torch.isnan(torch.view_as_real(S)).any()
        assert np.max(np.abs(S[:, cols].cpu().numpy() - fsv_route.unitary_columns(n, ops, cols))) <= 1e-6
    finally:
        B.tqs_circuit_destroy(c)
