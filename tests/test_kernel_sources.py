"""Rules of the kernel sources that no run can show reliably."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2010_14298_gb300", "csrc")


def _code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


def test_warp_operations_name_their_lanes():
    """__activemask() holds whichever lanes happen to be converged, which says
    nothing about which lanes will reach a shuffle: every warp operation gets
    its mask from the program (all lanes, or a ballot of all lanes)."""
    for name in sorted(os.listdir(CSRC)):
        assert "__activemask" not in _code(name), name
