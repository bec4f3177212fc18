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


def test_shared_memory_limits_do_not_follow_the_call():
    """A kernel's limit of dynamic shared memory is state that all threads
    share: set to one call's size, it refuses the launch of another thread
    whose blocks are larger.  One helper raises it, to a constant."""
    uses = []
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        uses += re.findall(r"cudaFuncSetAttribute\(([^;]*)\)", text)
    assert len(uses) == 1 and re.sub(r"\s+", " ", uses[0]).endswith(
        "cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_LIMIT")
