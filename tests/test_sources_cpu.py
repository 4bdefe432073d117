"""Rules on the sources that need no GPU."""
import glob
import os

from conftest import ROOT


def test_no_multicast_loads():
    """bench.py and multigpu.py run the library under several ranks, where TMA loads with cluster
    multicast are not used: no source has one, not even behind an option."""
    srcs = glob.glob(os.path.join(ROOT, "paper_2407_10205_gb300", "csrc", "*"))
    assert len(srcs) > 10
    for p in srcs:
        assert "multicast::cluster" not in open(p).read(), os.path.basename(p)
