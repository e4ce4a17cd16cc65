"""Sampling of batches whose states one CTA each samples: every number of
chunks a thread can own (1, 2, 4), states smaller than a chunk, mixed sizes in
one batch, fewer and more shots than threads, zero entries and a shot on either
side of every boundary.  Integer probabilities over a power of two make the
cumulative sums exact, so every index is determined."""
import numpy as np
import pytest

from paper_2305_14398_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def want(p, u):
    """First i with p_i > 0 and u T < C_i (exact: integers below 2^53)."""
    c = np.cumsum(p)
    return np.searchsorted(c, u * c[-1], side="right")


@pytest.mark.parametrize("ns", [[1], [2, 3], [3, 8, 5], [11, 4], [12, 12], [13, 1, 10]])
@pytest.mark.parametrize("shots", [1, 33, 700])
def test_batch_sample_exact(ns, shots):
    g = np.random.default_rng([99, shots, *ns])
    b = B.tqs_batch_create_packed(*B.pack_ops([(n, [("h", (0,), ())]) for n in ns]))
    try:
        ps, us, ws = [], [], []
        for n in ns:
            p = g.integers(0, 9, 1 << n) * (g.random(1 << n) < 0.7)
            p[int(g.integers(0, 1 << n))] += 1
            T = 1 << 20  # the total: a power of two, so u T is exact
            p[int(np.flatnonzero(p)[0])] += T - int(p.sum())
            u = g.integers(0, T, shots) / T  # on the boundaries C_i / T as often as between them
            ps.append(p / T)
            us.append(u)
            ws.append(want(p.astype(np.float64), u))
        probs = torch.from_numpy(np.concatenate(ps)).cuda()
        uu = torch.from_numpy(np.concatenate(us)).cuda()
        out = torch.full((len(ns) * shots,), -7, dtype=torch.int64, device="cuda")
        B.tqs_batch_sample(b, probs, shots, uu, out)
        assert np.array_equal(out.cpu().numpy(), np.concatenate(ws))
        zeros = torch.zeros_like(probs)
        B.tqs_batch_sample(b, zeros, shots, uu, out)
        assert torch.all(out == -1)
    finally:
        B.tqs_batch_destroy(b)
