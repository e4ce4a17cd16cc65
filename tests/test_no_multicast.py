"""The library runs on one GPU or, a process each, on several; its sources hold no
multicast load or arrival, not even behind an option."""
import glob
import os

import paper_2305_14398_gb300 as pkg


def test_no_multicast_in_the_kernels():
    files = glob.glob(os.path.join(os.path.dirname(pkg.__file__), "csrc", "*"))
    assert len(files) > 10
    for f in files:
        with open(f) as h:
            assert "multicast::cluster" not in h.read(), f
