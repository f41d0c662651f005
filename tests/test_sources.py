"""What the library's sources may not name."""
import glob
import os

import __graft_entry__ as ge


def test_no_multicast_loads():
    """Ranks of a sharded screen run the same kernels as one GPU: none of them delivers a copy to several CTAs."""
    files = glob.glob(os.path.join(ge.ROOT, "paper_2602_06986_gb300", "csrc", "*.cu*"))
    assert files
    assert not [f for f in files if "multicast" in open(f).read()]
