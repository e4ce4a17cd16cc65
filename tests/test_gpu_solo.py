"""A single circuit of up to 11 qubits takes a CTA of its own (a thread per
group); its states, probabilities and norm are bitwise those of the same
circuit in a batch, for both widths of the warp class, from a basis state and
from a given one."""
import numpy as np
import pytest

from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("team_warps", [1, 2])
@pytest.mark.parametrize("n", list(range(1, 12)))
def test_single_equals_batch(n, team_warps):
    q = max(4, n)
    old = B.tqs_get_option(B.OPT_TEAM_WARPS, q)
    B.tqs_set_option(B.OPT_TEAM_WARPS, q, team_warps)
    try:
        for ops in (W.qft_on_basis(n, (1 << n) - 1), W.random_small(n, 5 * n, (98, n))):
            c = B.circuit_from_ops(n, ops)
            b = B.tqs_batch_create([c, c])
            try:
                one = [torch.empty(1 << n, dtype=d, device="cuda") for d in (torch.complex64, torch.float64)]
                two = [torch.empty(2 << n, dtype=d, device="cuda") for d in (torch.complex64, torch.float64)]
                norm, norms = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (1, 2))
                B.tqs_simulate(c, one[0], probs=one[1], norm=norm)
                B.tqs_batch_run(b, two[0], two[1], norms)
                for x, y in zip(one + [norm], two + [norms]):
                    m = x.numel()
                    assert torch.equal(x, y[:m]) and torch.equal(x, y[m:])
                init = torch.zeros_like(one[0])
                init[0] = 1.0
                again = torch.empty_like(init)
                B.tqs_simulate(c, again, init=init, norm=norm)
                assert np.max(np.abs((again - one[0]).cpu().numpy())) <= 1e-6
                assert abs(float(norm) - float(norms[0])) <= 1e-6
            finally:
                B.tqs_batch_destroy(b)
                B.tqs_circuit_destroy(c)
    finally:
        B.tqs_set_option(B.OPT_TEAM_WARPS, q, old)
