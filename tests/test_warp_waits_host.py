"""The tensor-core kernels' waits give one answer per warp.

field_wait() answers lane by lane, and what follows a wait in these kernels are
warp-wide instructions, so a warp whose lanes disagree on an expired wait would never
leave them.  A GPU cannot be made to show that safely; the source shows it: every wait
of a whole warp goes through warp_wait(), every look at the abort word through a vote,
and a bare field_wait() stands only where one lane waits alone."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_08146_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name,alone", [("sc_field_tensor.cu", 0), ("sc_idft.cu", 1)])
def test_waits_are_votes(name, alone):
    code = _code(name)
    assert "warp_wait(" in code
    bare = [m.start() for m in re.finditer(r"\bfield_wait\(", code)]
    assert len(bare) == alone
    for at in bare:  # the last enclosing condition before it is the single lane's
        assert code.rfind("if (lane == 0) {", 0, at) > code.rfind("__syncwarp", 0, at)
    # no condition reads the CTA's abort word but through a vote
    assert not re.findall(r"(?:if|while) \(!?\*s_abort", code)
