"""Cluster-multicast loads stay out of the library: bench.py runs it on several GPUs
at once (one replica each), where they are not to be used."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2112_10526_gb300", "csrc")


def test_no_kernel_multicasts():
    files = [f for ext in ("*.cu", "*.cuh", "*.h") for f in glob.glob(os.path.join(CSRC, ext))]
    assert files
    for f in files:
        assert "multicast" not in open(f).read(), f
