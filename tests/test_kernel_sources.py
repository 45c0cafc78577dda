"""What the kernels' sources leave out, because no run can show that it is absent."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1912_02868_gb300", "csrc")


def _code(path):
    """The source without its comments."""
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


def test_shuffles_name_their_lanes():
    # __activemask() is whatever lanes happen to run together: after a loop or branch that
    # differs by lane, a shuffle over it may leave out lanes that it should read
    files = glob.glob(os.path.join(CSRC, "*.cu*"))
    assert files and not [os.path.basename(f) for f in files if "__activemask" in _code(f)]
