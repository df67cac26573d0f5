"""Rules that the kernel sources keep, read from their text (no GPU)."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2607_00790_gb300", "csrc")


def sources():
    files = sorted(f for e in ("*.cu", "*.cuh", "*.h") for f in glob.glob(os.path.join(CSRC, e)))
    assert files
    return {os.path.basename(f): open(f).read() for f in files}


def test_no_multicast():
    """A CTA loads and releases its own tiles only: one process per GPU runs this library, and an arrival
    at another CTA's barrier could come after that CTA has left."""
    assert [f for f, s in sources().items() if "multicast" in s] == []
