"""What the library's sources may not hold."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09338_gb300", "csrc")


def test_no_multicast_loads():
    """Programs on several GPUs load the library too: every CTA loads its own tiles, no copy is multicast to a cluster."""
    files = glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h"))
    assert len(files) > 10
    for f in files:
        with open(f) as fh:
            assert ".multicast::cluster" not in fh.read(), os.path.basename(f)
