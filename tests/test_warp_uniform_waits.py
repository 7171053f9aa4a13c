"""Bounded waits give up as whole warps.  Lanes that give up alone go on to the block's barrier while the others stand in
an instruction that needs the whole warp (tcgen05.ld, elect.sync, __syncwarp) and has no limit.  On the GPU the
difference would be a hang, so the sources are looked at instead."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_19867_b200", "csrc")


def _statements(name):
    text = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
    return [" ".join(s.split()) for s in re.split(r"[;{}]", text)]


@pytest.mark.parametrize("name", sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh"))))
def test_every_wait_is_voted_on(name):
    statements = _statements(name)
    for this, following in zip(statements, statements[1:] + [""]):
        if "__device__" in this:                                    # a definition
            continue
        # the waits of single lanes: the loop behind wait_warp's first try, and the wait for a counter
        for call in re.finditer(r"\b(wait_slow|wait_counter)\(", this):
            voted = this[:call.start()].endswith("__all_sync(0xffffffffu, ")
            result = re.search(r"(\w+) = $", this[:call.start()])   # voted on by the next statement
            later = result and following == f"{result[1]} = __all_sync(0xffffffffu, {result[1]})"
            assert voted or later, this
        if name != "wfq_ptx.cuh":
            assert "mbar_try_wait(" not in this, this


def test_wait_warp_votes_on_both_tries():
    body = " ".join(_statements("wfq_ptx.cuh"))
    body = body[body.index("bool wait_warp("):body.index("void drain(")]
    assert len(re.findall(r"__all_sync\(0xffffffffu, (ptx::mbar_try_wait|wait_slow)\(", body)) == 2
