"""Batch sampling on either side of the numbers of shots at which its blocks grow."""
import pytest

from test_gpu_sample_small import test_batch_sample_exact as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shots", [64, 65, 128, 129, 512, 513])
@pytest.mark.parametrize("ns", [[1], [6, 3], [10]])
def test_shots_at_the_edges(ns, shots):
    check(ns, shots)
