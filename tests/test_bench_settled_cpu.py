"""bench.py without a GPU: the smoother's bytes when launches visited settled
tiles only."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_smooth_bytes_are_those_of_the_visited_tiles():
    """Where launches visited a part of the nodes, the class's bytes count and
    not launches times a plain launch."""
    sys.path.insert(0, ROOT)
    import bench
    from paper_0710_0736_gb300 import ac
    k = ac.PROF_CLASSES.index("smooth")
    p = ac.ac_profile()
    p.launches[k], p.smooth_bytes_per_launch = 12, 1000.0
    p.smooth_corr_launches, p.smooth_corr_extra_bytes = 2, 250.0
    p.bytes[k] = 430.0
    assert bench.smooth_bytes(p) == 430.0
