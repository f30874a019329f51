"""A bounded wait gives up lane by lane: the first lane that finds the abort
flag set leaves it while another may still find its barrier complete.  Where a
warp goes on to warp-wide operations after a wait, its lanes must take one
answer (mbar_wait_warp), or an aborted launch would leave some of them in a
collective that the others never reach.  Checked on the sources of the kernels
whose warps wait as a whole: a wait of single lanes stands only where one lane
runs the loop, in the list below."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2608_23805_gb300", "csrc")

# the waits of a single lane, or of lanes that meet no collective before the
# kernel's closing barrier: (a barrier's name) in each file
SINGLE = {
    "gemm_cols.cu": ["sempty",   # bf16 weight producer, lane 0
                     "wempty",   # 4-bit weight producer: copies only
                     "never"],   # the injected stall, thread 0
    "router_tc.cu": ["empty",    # x producer, lane 0
                     "never"],
}


@pytest.mark.parametrize("name", sorted(SINGLE))
def test_waits_before_collectives_are_of_the_whole_warp(name):
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    # __all_sync(..., mbar_wait(..)) is a wait of the warp, as in mbar_wait_warp
    waits = [m.group(2) for m in re.finditer(r"(__all_sync\(0xffffffffu, )?\bmbar_wait\(&?(\w+)", text)
             if not m.group(1)]
    assert sorted(waits) == sorted(SINGLE[name])
