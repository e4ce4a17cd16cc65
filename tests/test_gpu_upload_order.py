"""A program's upload does not depend on host memory that a later call reuses:
circuits simulated one after the other while the stream is busy, with the
page-locked buffers of a destroyed batch in the pool, give the bits of the same
circuits simulated with a wait after each."""
import pytest

from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def run_all(circs, call, busy):
    handles = [B.circuit_from_ops(n, ops) for n, ops in circs]
    outs = [torch.zeros(1 << n, dtype=torch.complex64, device="cuda") for n, _ in circs]
    try:
        torch.cuda.synchronize()
        if busy is not None:
            for _ in range(20):
                busy @ busy
        for h, o in zip(handles, outs):
            call(h, o)
            if busy is None:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
    finally:
        for h in handles:
            B.tqs_circuit_destroy(h)
    return outs


@pytest.mark.parametrize("sizes", [(9, 10, 11), (12, 14, 16)])
def test_lone_circuits_on_a_busy_stream(sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pool = [B.circuit_from_ops(10, W.random_mixed(10, 20, (51, i))) for i in range(20)]
    b = B.tqs_batch_create(pool * 20)
    st = torch.empty(400 << 10, dtype=torch.complex64, device="cuda")
    B.tqs_batch_run(b, st, None, None)
    torch.cuda.synchronize()
    B.tqs_batch_destroy(b)
    for c in pool:
        B.tqs_circuit_destroy(c)
    circs = [(n, W.random_mixed(n, 8, (52, n, i))) for i in range(8) for n in sizes]
    want = run_all(circs, B.tqs_simulate, None)
    got = run_all(circs, B.tqs_simulate, torch.ones(8192, 8192, device="cuda"))
    for x, y in zip(want, got):
        assert torch.equal(x, y)
