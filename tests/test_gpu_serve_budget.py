"""The block sums of cooperating CTAs count against a server's memory budget:
with room they are part of the bytes held, and a budget of exactly one request
still serves it, bitwise the same, on one CTA."""
import re
import time

import numpy as np
import pytest

from paper_2305_14398_gb300 import binding as B
from paper_2305_14398_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def serve_one(budget, n, packed):
    sv = B.tqs_server_create(budget, 1, 1)
    try:
        B.tqs_server_submit_packed(sv, 0, n, packed)
        end = time.monotonic() + 30
        while len(B.tqs_server_poll(sv)) == 0:
            assert time.monotonic() < end
        st, nm = B.tqs_server_take(sv, 0, n)
        return st, nm, B.tqs_server_stats(sv)
    finally:
        B.tqs_server_destroy(sv)


@pytest.mark.parametrize("n", [15, 16])
def test_block_sums_in_budget(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    packed = B.pack_request(W.random_layered(n, 3, (17, n)))
    with pytest.raises(Exception, match="needs") as refused:
        serve_one(1, n, packed)
    need = int(re.search(r"needs (\d+) bytes", str(refused.value)).group(1))
    wide_st, wide_nm, wide = serve_one(1 << 30, n, packed)
    tight_st, tight_nm, tight = serve_one(need, n, packed)
    assert wide["peak_bytes"] == need + 4 * (1 << 16) // 16
    assert tight["peak_bytes"] == need
    assert wide["bytes_in_use"] == tight["bytes_in_use"] == 0
    assert np.array_equal(wide_st.view(np.uint32), tight_st.view(np.uint32))
    assert wide_nm == tight_nm
