"""Dense step matrices by row expansion (n >= 10) at the edges of its blocks: two
rows to a block or one, two-qubit factors whose partner lies among the last
three qubits, below them or among the lowest, custom factors across all of
them, idle qubits.  Sampled columns against the oracle's, 1e-6 (products of at
most n FP32 entries)."""
import numpy as np
import pytest

from oracle import fsv_route
from oracle import gates as G
from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W
from test_host_program import rand_unitary

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def steps(n):
    t, m = n - 1, n - 4
    yield [("cu", (t, 0), W.random_small(2, 1, (97, n), names=("cu",))[0][2]), ("cp", (1, m), (0.4,)),
           ("swap", (t - 1, t - 2), ()), ("u3", (2,), (0.3, 0.2, 0.1))]
    yield [("cx", (0, t), ()), ("cu", (t - 1, m), W.random_small(2, 1, (98, n), names=("cu",))[0][2]),
           ("rx", (t - 2,), (1.1,))]
    yield [("unitary", (t, 0, m), G.custom_params(rand_unitary(3, n))),
           ("unitary", (t - 2, 1, t - 1, 2, 3), G.custom_params(rand_unitary(5, n)))]
    yield [("h", (q,), ()) for q in range(n)]


@pytest.mark.parametrize("n", [9, 10, 11, 12, 13, 14])
def test_step_matrix_columns(n):
    S = torch.empty((1 << n, 1 << n), dtype=torch.complex64, device="cuda")
    cols = sorted({0, 1, (1 << n) - 1, 1 << (n - 3), 5 * 41 + 7, (1 << n) - 6})
    for ops in steps(n):
        c = B.circuit_from_ops(n, ops)
        try:
            S.fill_(float("nan"))
            B.tqs_materialize_step(c, 0, S)
            assert not torch.isnan(torch.view_as_real(S)).any()
            got = S[:, cols].cpu().numpy()
            assert np.max(np.abs(got - fsv_route.unitary_columns(n, ops, cols))) <= 1e-6
        finally:
            B.tqs_circuit_destroy(c)
