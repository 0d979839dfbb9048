"""The stalls of the spans and the two-row stencil are host state only."""
import pytest

import paper_1603_03971_gb300 as rtm
from paper_1603_03971_gb300 import _lib


def test_every_stall_kernel_arms_and_disarms():
    for kernel in (rtm.STALL_STENCIL, rtm.STALL_ENCODER, rtm.STALL_ROWS, rtm.STALL_SPAN):
        rtm.set_test_stall(kernel, 0)
        rtm.set_test_stall(kernel, -1)
    with pytest.raises(_lib.RtmError):
        rtm.set_test_stall(rtm.STALL_SPAN + 1, 0)
