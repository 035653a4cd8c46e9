"""CPU check of the kernel sources: the one library is loaded by every rank of a multi-rank run, and a
TMA load with cluster multicast is not for code that several GPUs run."""
import glob
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_multicast_load():
    files = glob.glob(os.path.join(ROOT, "paper_2509_06856_gb300", "csrc", "*.cu*"))
    assert files
    for f in files:
        assert ".multicast::" not in open(f).read(), f
