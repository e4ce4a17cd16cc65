"""A lone 14-qubit circuit with general gates and 8 passes or more runs on
cooperating CTAs (tqs_simulate); with the option at 1, and in a batch, on one
CTA: the same states, probabilities and norm, bit for bit."""
import pytest
import torch

from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W

pytestmark = pytest.mark.gpu
N = 14


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("layers", [4, 10])
def test_cooperating_ctas_at_14_qubits(layers, threads):
    c = B.circuit_from_ops(N, W.random_layered(N, layers, (97, N, layers)))
    old = B.tqs_get_option(B.OPT_CTA_THREADS, 0)
    B.tqs_set_option(B.OPT_CTA_THREADS, 0, threads)
    b = B.tqs_batch_create([c, c])
    try:
        passes, ops = B.tqs_circuit_program(c)[:2]
        # what the cooperating CTAs ask for: else every run below is the same one
        assert len(passes) >= 8 and any(32 <= int(k) < 36 for k in ops["code"])
        got = []
        for ctas in (8, 2, 1):
            B.tqs_set_option(B.OPT_MULTI_CTAS, 0, ctas)
            out = torch.empty(1 << N, dtype=torch.complex64, device="cuda")
            pr = torch.empty(1 << N, dtype=torch.float64, device="cuda")
            nm = torch.empty(1, dtype=torch.float64, device="cuda")
            B.tqs_simulate(c, out, probs=pr, norm=nm)
            got.append((out, pr, nm))
        st = torch.empty(2 << N, dtype=torch.complex64, device="cuda")
        pr = torch.empty(2 << N, dtype=torch.float64, device="cuda")
        nm = torch.empty(2, dtype=torch.float64, device="cuda")
        B.tqs_batch_run(b, st, probs=pr, norms=nm)
        got += [(st[k << N:(k + 1) << N], pr[k << N:(k + 1) << N], nm[k:k + 1]) for k in range(2)]
        for other in got[1:]:
            assert all(torch.equal(x, y) for x, y in zip(got[0], other))
        assert abs(float(got[0][2]) - 1.0) <= 1e-6
    finally:
        B.tqs_set_option(B.OPT_MULTI_CTAS, 0, 8)
        B.tqs_set_option(B.OPT_CTA_THREADS, 0, old)
        B.tqs_batch_destroy(b)
        B.tqs_circuit_destroy(c)
