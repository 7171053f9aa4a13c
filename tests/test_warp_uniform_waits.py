"""Bounded waits of the warp-specialised kernels: a role gives up as a whole warp.  Lanes that give up alone go on to the
block's barrier while the others stand in an instruction that needs the whole warp (tcgen05.ld, elect.sync, __syncwarp)
and has no limit.  On the GPU the difference would be a hang, so the sources are looked at instead."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_19867_b200", "csrc")


def _statements(path):
    text = re.sub(r"/\*.*?\*/|//[^\n]*", "", open(path).read(), flags=re.S)
    return [" ".join(s.split()) for s in re.split(r"[;{}]", text)]


@pytest.mark.parametrize("name", ["wfq_gemm.cu", "wfq_input_transform_tc.cu", "wfq_input_transform_tcn.cu"])
def test_every_wait_is_voted_on(name):
    found = 0
    statements = _statements(os.path.join(CSRC, name))
    for this, following in zip(statements, statements[1:] + [""]):
        if "__device__" in this:                                    # a definition
            continue
        for call in re.finditer(r"\bwait_(bounded|counter)\(", this):
            found += 1
            voted = this[:call.start()].endswith("__all_sync(0xffffffffu, ")
            unused = call.start() == 0                              # nothing depends on the result
            result = re.search(r"(\w+) = $", this[:call.start()])   # voted on by the next statement
            later = result and following == f"{result[1]} = __all_sync(0xffffffffu, {result[1]})"
            assert voted or unused or later, this
    assert found >= 4
