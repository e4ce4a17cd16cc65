"""The tensor-core chain multiplies consecutive steps whose gates fall into blocks
of at most 5 qubits before it forms products: circuits that end in one run
(no product at all), blocks grown to the limit by every gate kind, gates that
wait for a later run, custom gates inside a block.  1e-4 against the oracle,
the chain's tolerance (1e-6 where no product is formed)."""
import numpy as np
import pytest

from oracle import fsv_route
from oracle import gates as G
from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W
from test_host_program import rand_unitary

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def within(n, qubits, count, seed):
    """Random gates of every kind on some qubits of n."""
    return [(name, tuple(qubits[q] for q in qs), ps)
            for name, qs, ps in W.random_small(len(qubits), count, (101, n, seed))]


def cases(n):
    yield "one run", within(n, [0, 2, 3, n - 1, 5], 30, 1) + within(n, [1, 4], 9, 2), 1e-6
    yield "every kind", list(W.random_small(n, 10 * n, (102, n))), 1e-4
    custom = [("unitary", (n - 1, 1, 3), G.custom_params(rand_unitary(3, n))),
              ("unitary", (4, 0, 2, 5, 6), G.custom_params(rand_unitary(5, n)))]
    yield "custom", (within(n, [0, 1, n - 1], 6, 3) + custom[:1] + within(n, [1, 3], 4, 4) + custom[1:] +
                     within(n, list(range(n)), 12, 5)), 1e-4
    yield "waiting", [("cx", (q, q + 1), ()) for q in range(n - 1)] + [("rx", (q,), (0.1 * q + 0.2,)) for q in range(n)] + [
        ("cp", (n - 1 - q, 0), (0.3 * q,)) for q in range(n - 1)], 1e-4


@pytest.mark.parametrize("prec", [B.PREC_TC_BF16X3, B.PREC_TC_TF32X3])
@pytest.mark.parametrize("n", [7, 9, 11])
def test_chain_of_runs(n, prec):
    cols = [0, 1, (1 << n) - 1, 77]
    for name, ops, tol in cases(n):
        c = B.circuit_from_ops(n, ops)
        try:
            U = torch.full((1 << n, 1 << n), float("nan"), dtype=torch.complex64, device="cuda")
            B.tqs_circuit_unitary(c, prec, U)
            got = U[:, cols].cpu().numpy()
            assert np.max(np.abs(got - fsv_route.unitary_columns(n, ops, cols))) <= tol, name
            part = torch.empty((1 << n, 128), dtype=torch.complex64, device="cuda")
            B.tqs_circuit_unitary_cols(c, prec, 0, 128, part)
            assert torch.equal(torch.view_as_real(part), torch.view_as_real(U[:, :128].contiguous())), name
        finally:
            B.tqs_circuit_destroy(c)
