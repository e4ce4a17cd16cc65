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


@pytest.mark.parametrize("count", [3, 1300, 2500])
def test_batches_on_either_team_equal_singles(count):
    """Batches on both sides of the rules that give circuits of the warp class a
    CTA each: with and without general gates, 8 to 11 qubits, more circuits
    than CTAs, instructions and custom unitaries (which stay on warps) between
    them; every copy bitwise the single call's."""
    from test_host_program import with_customs
    g = W.rng(97)
    kinds = [(n, ops) for n in (5, 9, 10, 11) for ops in (W.qft_on_basis(n, 3), W.random_mixed(n, 5, (97, n)))]
    extra = [(10, [("h", (0,), ()), ("measure", (0,), ()), ("rx", (1,), (0.3,))]), (9, with_customs(9, 7)[0])]
    circs = extra + [kinds[int(g.integers(0, len(kinds)))] for _ in range(count)]
    handles = {}
    for n, ops in circs:
        if id(ops) not in handles:
            handles[id(ops)] = B.circuit_from_ops(n, ops)
    try:
        b = B.tqs_batch_create([handles[id(ops)] for _, ops in circs])
        try:
            _, total, offs = B.tqs_batch_info(b)
            st = torch.empty(total, dtype=torch.complex64, device="cuda")
            pr = torch.empty(total, dtype=torch.float64, device="cuda")
            nm = torch.empty(len(circs), dtype=torch.float64, device="cuda")
            u = torch.full((1,), 0.25, dtype=torch.float64, device="cuda")
            B.tqs_batch_run_measured(b, st, u, probs=pr, norms=nm)
            assert B.tqs_batch_launch_info(b, 0)["jobs"] == len(circs)
        finally:
            B.tqs_batch_destroy(b)
        single = {}
        for n, ops in circs:
            if id(ops) in single:
                continue
            o = [torch.empty(1 << n, dtype=d, device="cuda") for d in (torch.complex64, torch.float64)]
            o.append(torch.empty(1, dtype=torch.float64, device="cuda"))
            B.tqs_simulate_measured(handles[id(ops)], o[0], u=u, probs=o[1], norm=o[2])
            single[id(ops)] = o
        for i, (n, ops) in enumerate(circs):
            s, p, m = single[id(ops)]
            assert torch.equal(st[offs[i]:offs[i + 1]], s) and torch.equal(pr[offs[i]:offs[i + 1]], p)
            assert float(nm[i]) == float(m)
    finally:
        for c in handles.values():
            B.tqs_circuit_destroy(c)


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("name", ["qft", "layered"])
def test_one_circuit_of_14_qubits_on_either_team(name, threads):
    """A lone 14-qubit circuit with general gates runs on cooperating CTAs, any
    other (and every one with the option at 1) on one: the same bits."""
    n = 14
    c = B.circuit_from_ops(n, W.qft_on_basis(n, 77) if name == "qft" else W.random_layered(n, 3, (98, n)))
    got = []
    old = B.tqs_get_option(B.OPT_CTA_THREADS, 0)
    B.tqs_set_option(B.OPT_CTA_THREADS, 0, threads)
    try:
        for k in (8, 3, 1):
            B.tqs_set_option(B.OPT_MULTI_CTAS, 0, k)
            out = torch.empty(1 << n, dtype=torch.complex64, device="cuda")
            pr = torch.empty(1 << n, dtype=torch.float64, device="cuda")
            nm = torch.empty(1, dtype=torch.float64, device="cuda")
            B.tqs_simulate(c, out, probs=pr, norm=nm)
            got.append((out, pr, nm))
        for other in got[1:]:
            assert all(torch.equal(x, y) for x, y in zip(got[0], other))
    finally:
        B.tqs_set_option(B.OPT_MULTI_CTAS, 0, 8)
        B.tqs_set_option(B.OPT_CTA_THREADS, 0, old)
        B.tqs_circuit_destroy(c)
