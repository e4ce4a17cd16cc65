"""Two host threads that launch the same kernels with different amounts of
shared memory: neither's launch fails for the other's (a kernel's limit is set
once, to all that the device has)."""
import threading

import pytest

from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def in_threads(works, rounds):
    errors = []

    def loop(work):
        try:
            for _ in range(rounds):
                work()
        except Exception as e:  # noqa: BLE001
            errors.append(repr(e))

    ts = [threading.Thread(target=loop, args=(w,)) for w in works]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert errors == []


def test_simulate_sizes_side_by_side():
    sizes = (13, 14, 13, 14)  # one CTA each: 64 and 128 KiB
    circuits = [B.circuit_from_ops(n, W.qft_on_basis(n, 5)) for n in sizes]
    streams = [torch.cuda.Stream() for _ in sizes]
    outs = [torch.empty(1 << n, dtype=torch.complex64, device="cuda") for n in sizes]
    wants = [torch.empty_like(o) for o in outs]
    try:
        for c, w in zip(circuits, wants):
            B.tqs_simulate(c, w)
        torch.cuda.synchronize()
        in_threads([lambda c=c, o=o, s=s: B.tqs_simulate(c, o, stream=s.cuda_stream)
                    for c, o, s in zip(circuits, outs, streams)], 3000)
        assert all(torch.equal(o, w) for o, w in zip(outs, wants))
    finally:
        for c in circuits:
            B.tqs_circuit_destroy(c)


def test_sample_sizes_side_by_side():
    sizes, shots = (3, 11, 3, 11), 200
    circuits = [B.circuit_from_ops(n, [("h", (q,), ()) for q in range(n)]) for n in sizes]
    batches = [B.tqs_batch_create([c] * 4) for c in circuits]
    streams = [torch.cuda.Stream() for _ in sizes]
    probs = [torch.full((4 << n,), 1.0 / (1 << n), dtype=torch.float64, device="cuda") for n in sizes]
    us = [torch.rand(4 * shots, dtype=torch.float64, device="cuda") for _ in sizes]
    outs = [torch.empty(4 * shots, dtype=torch.int64, device="cuda") for _ in sizes]
    wants = [torch.empty_like(o) for o in outs]
    try:
        for b, p, u, w in zip(batches, probs, us, wants):
            B.tqs_batch_sample(b, p, shots, u, w)
        torch.cuda.synchronize()
        in_threads([lambda b=b, p=p, u=u, o=o, s=s: B.tqs_batch_sample(b, p, shots, u, o, stream=s.cuda_stream)
                    for b, p, u, o, s in zip(batches, probs, us, outs, streams)], 3000)
        assert all(torch.equal(o, w) for o, w in zip(outs, wants))
    finally:
        for b in batches:
            B.tqs_batch_destroy(b)
        for c in circuits:
            B.tqs_circuit_destroy(c)
