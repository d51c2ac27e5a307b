"""Bounded waits that warp-wide instructions follow: a warp gives up as one,
whichever of its lanes run out of polls."""
import ctypes
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_28183_gb300", "csrc")


@pytest.mark.gpu
@pytest.mark.parametrize("gave_up", [0, 1, 16, 31, 32])
def test_warp_gives_up_as_one(gave_up):
    from paper_2608_28183_gb300 import build, nlos
    build.build()
    n = ctypes.c_int(-1)
    assert nlos.load_library().nlos_selftest_warp_wait(gave_up, ctypes.byref(n)) == 0
    assert n.value == (0 if gave_up else 32)


def test_depth_sum_warps_wait_as_one():
    """In the pipelined depth sum, the waits of whole warps (epilogue,
    builders) come before tcgen05.ld and __syncwarp."""
    text = open(os.path.join(CSRC, "pf_umma.cu")).read()
    epilogue = text[text.index("} else if (warp >= kEpiWarp0) {"):text.index("if (warp == kMmaWarp) tmem_dealloc(tm, 2")]
    assert len(re.findall(r"mbar_wait_warp\(", epilogue)) == 2
    assert "mbar_wait_bounded(" not in epilogue
