"""No warp of a kernel with bounded waits waits without a limit for one that may have given up.

A warp whose wait on an mbarrier runs out leaves its loop for the teardown; a named barrier (bar.sync) behind such a wait is
then one arrival short and has no limit of its own.  Read from the sources: stalling a GPU to see it is not an option."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_17419_b200", "csrc")


# (the first-order kernel's barrier 6 lies behind its loop: each of the three warps comes to it, having given up or not)
@pytest.mark.parametrize("name,fine", [("kata_tc_attend.cu", ""), ("kata_tc_state.cu", ""), ("kata_tc_bwd.cu", ""),
                                       ("kata_tc_stream.cu", ""), ("kata_tc_order1.cu", "bar.sync 6, 96")])
def test_named_barriers_come_before_bounded_waits(name, fine):
    text = open(os.path.join(CSRC, name)).read()
    kernel = re.search(r"__global__ void __launch_bounds__.*?// -{16} (teardown|end of the pass)", text, flags=re.S).group(0)
    roles = re.split(r"\n\s*// =+ ", kernel)                  # the banners of the warps' roles
    assert len(roles) >= 5
    for role in roles:
        for barrier in re.finditer(r"\b(bar|barrier)\.(cta\.)?(sync|red)|named_barrier", role):
            if not (fine and role.startswith(fine, barrier.start())):
                assert "wait_or_abort" not in role[:barrier.start()], role[:60]
