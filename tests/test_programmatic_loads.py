"""Loads of the kernels that are launched programmatically.  Such a kernel runs before its predecessor in the stream has
ended, so what the predecessor writes must not be read through the read-only path (`__ldg`, `ld.global.nc`): that path is
for data nobody writes while the kernel runs, and its loads may be moved above the wait.  Every `__ldg` in these files is
of a named operand that was complete before the predecessor began."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_01216_gb300", "csrc")

COMPLETE = {
    # the forward activations (masks of the backward pass, the head's input), whose kernels ended several launches ago
    "unet.cu": ["vox(s, ", "reinterpret_cast<const uint4*>(Hd "],
    # the mask likewise, and the caller's input (the first kernel of a call is launched as usual)
    "unet_conv.cu": ["reinterpret_cast<const uint4*>(\n                    a.mask ", "a.hx + gi"],
}


def code(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


@pytest.mark.parametrize("name", sorted(COMPLETE))
def test_read_only_loads_are_of_complete_operands(name):
    src = code(name)
    loads = [src[m.end():m.end() + 90] for m in re.finditer(r"__ldg\(", src)]
    assert loads
    for arg in loads:
        assert any(arg.startswith(ok) for ok in COMPLETE[name]), (name, arg)
    assert "ld.global.nc" not in src
