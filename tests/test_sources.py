"""What the device sources must not say."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1503_00638_gb300", "csrc")


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))),
                         ids=lambda p: os.path.basename(p))
def test_warp_collectives_name_lanes_known_beforehand(path):
    """The lanes that __activemask() reports need not be together any more at
    the next instruction, so it is no mask for a collective."""
    text = re.sub(r"//[^\n]*", "", open(path).read())
    assert "__activemask" not in text
