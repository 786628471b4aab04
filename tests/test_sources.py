"""What the CUDA sources may not hold."""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_copy_goes_to_several_ctas():
    """The library also runs as one process per GPU, where bulk copies into several CTAs of a cluster
    are not used (commits that arrive on several CTAs' barriers are no copies)."""
    files = glob.glob(os.path.join(ROOT, "paper_2205_01435_gb300", "csrc", "*.cu*"))
    assert files
    for f in files:
        for n, line in enumerate(open(f), 1):
            assert not re.search(r"cp\.async\.bulk.*multi" + "cast", line), f"{f}:{n}"
