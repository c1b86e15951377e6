"""The library issues no TMA multicast load and no multicast commit: the same kernels run in jobs of several
GPUs. Read from the sources; needs no GPU."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_00391_gb300", "csrc")


def test_no_multicast_in_the_sources():
    files = glob.glob(os.path.join(CSRC, "*.cu*"))
    assert len(files) >= 10
    assert not [f for f in files if ".multicast::" in open(f).read()]
