"""Statements about the kernels' sources."""
import glob
import os

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2111_07347_gb300", "csrc")


def test_no_multicast_loads():
    """Contexts of several GPUs run the same kernels (one process per GPU), so none of them issues a
    multicast copy or arrival."""
    files = glob.glob(os.path.join(CSRC, "*"))
    assert len(files) > 10
    for f in files:
        with open(f, encoding="utf-8") as fh:
            assert "multicast" not in fh.read(), f
