"""Batches launch the circuits of 12, 13 and 14 qubits separately, the smaller
with fewer threads than the team whose norm they form: states, probabilities
and norms are bitwise those of single calls and of batches of any mixture and
number, for both thread counts of the option, with and without instructions."""
import pytest

from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def batch(circs, reps):
    b = B.tqs_batch_create_packed(*B.pack_ops(circs * reps))
    try:
        count, total, offs = B.tqs_batch_info(b)
        st = torch.empty(total, dtype=torch.complex64, device="cuda")
        pr = torch.empty(total, dtype=torch.float64, device="cuda")
        nm = torch.empty(count, dtype=torch.float64, device="cuda")
        B.tqs_batch_run(b, st, pr, nm)
        info = B.tqs_batch_launch_info(b, 1)
        assert info["jobs"] == sum(n >= 12 for n, _ in circs) * reps
        return [(st[offs[i]:offs[i + 1]], pr[offs[i]:offs[i + 1]], nm[i]) for i in range(count)]
    finally:
        B.tqs_batch_destroy(b)


@pytest.mark.parametrize("threads", [256, 512])
def test_sizes_apart_same_bits(threads):
    circs = [(n, ops) for n in (12, 13, 14, 7) for ops in (W.qft_on_basis(n, 5), W.random_mixed(n, 6, (99, n)))]
    old = B.tqs_get_option(B.OPT_CTA_THREADS, 0)
    B.tqs_set_option(B.OPT_CTA_THREADS, 0, threads)
    try:
        few, many = batch(circs, 1), batch(circs, 40)  # 80 circuits of 13 qubits; then more than one per SM
        crowd = batch([c for c in circs if c[0] == 13], 90)
        for i, (n, ops) in enumerate(circs):
            c = B.circuit_from_ops(n, ops)
            try:
                st = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
                pr = torch.empty(1 << n, dtype=torch.float64, device="cuda")
                nm = torch.empty(1, dtype=torch.float64, device="cuda")
                B.tqs_simulate(c, st, probs=pr, norm=nm)
            finally:
                B.tqs_circuit_destroy(c)
            others = [few[i], many[i], many[-len(circs) + i]] + ([crowd[i - 2]] if n == 13 else [])
            for s, p, m in others:
                assert torch.equal(s, st) and torch.equal(p, pr) and float(m) == float(nm)
    finally:
        B.tqs_set_option(B.OPT_CTA_THREADS, 0, old)
