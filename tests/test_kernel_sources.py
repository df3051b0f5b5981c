"""Rules of the kernels' sources that a run on the GPU cannot show: breaking one gives a wrong sum or a hang
only when warps happen to be scheduled badly, so the sources themselves are read (no GPU needed)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_13846_gb300", "csrc")


def _source(name):
    """A source file without its comments."""
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))


def test_warp_collectives_name_their_lanes():
    """No collective takes the lanes that happen to be converged for the lanes that take part."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert "__activemask" not in _source(os.path.basename(path)), path
