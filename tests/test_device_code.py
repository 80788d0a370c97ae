"""Rules the device code keeps that no run on one GPU can show to hold."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_14172_gb300", "csrc")


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_warp_operations_name_their_lanes(name):
    """__activemask() gives the lanes that happen to run together and brings
    none together: a shuffle over it may read a lane that is not there.  Every
    warp operation names the lanes it needs instead."""
    src = open(os.path.join(CSRC, name)).read()
    code = re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)
    assert "__activemask" not in code
