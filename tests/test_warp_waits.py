"""The waits of whole warps in the tensor-core kernels: one verdict for all lanes, whichever lane's wait runs out."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_07006_gb300", "csrc")


def test_kernels_wait_through_the_voting_form():
    """mbar_spin gives each lane a verdict of its own; a warp that branches on it may meet elect.sync in pieces."""
    for name in sorted(os.listdir(CSRC)):
        if name != "ptx_sm100.cuh":
            with open(os.path.join(CSRC, name)) as f:
                assert not re.search(r"\bmbar_spin\s*\(", f.read()), name


@pytest.mark.gpu
def test_a_wait_that_runs_out_in_some_lanes_runs_out_in_all():
    from paper_2304_07006_gb300 import Context
    with Context("fp16x2") as c:
        assert c.selftest_wait_timeout(20) == -6      # XTC_ERR_TIMEOUT; 0 where the lanes disagree
