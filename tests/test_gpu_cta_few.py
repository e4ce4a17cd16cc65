"""Circuits of 12 and 13 qubits without general gates: few take all the threads
of a CTA, many half of them; the same states, probabilities and norms."""
import pytest

from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [12, 13])
def test_few_and_many_programs(n):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    c = B.circuit_from_ops(n, W.qft_on_basis(n, 77))
    got = []
    try:
        for count in (2, 2 * sms, 2 * sms + 1):
            b = B.tqs_batch_create([c] * count)
            try:
                st = torch.empty(count << n, dtype=torch.complex64, device="cuda")
                pr = torch.empty(count << n, dtype=torch.float64, device="cuda")
                nm = torch.empty(count, dtype=torch.float64, device="cuda")
                B.tqs_batch_run(b, st, probs=pr, norms=nm)
                assert B.tqs_batch_launch_info(b, 1)["threads"] == (256 if count > 2 * sms else 512)
                for k in (0, count - 1):
                    got.append((st[k << n:(k + 1) << n].clone(), pr[k << n:(k + 1) << n].clone(), nm[k:k + 1].clone()))
            finally:
                B.tqs_batch_destroy(b)
        for other in got[1:]:
            assert all(torch.equal(x, y) for x, y in zip(got[0], other))
    finally:
        B.tqs_circuit_destroy(c)
