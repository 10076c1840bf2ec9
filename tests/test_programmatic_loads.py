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
    # the handle's tables and a plan's descriptors: fr3d_invert builds what changed before the transform
    "fft2d.cuh": ["tw_full + ", "a + s * N", "p + l", "p + 3 * l", "wp + e"],
    "fft_engine.cuh": ["tw_g + "],
    "fused.cuh": ["a.tw_n + ", "Aj + ", "a.bbin + ", "drow + ", "a.Dd + ", "wq + "],
    "inv_queue.cu": ["a.tw_n + ", "Aj + ", "a.bbin + ", "a.Dd + ", "&ql.tab["],
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
    # the queue streams the combination weights (a table) through the read-only path
    assert src.count("ld.global.nc") == (1 if name == "inv_queue.cu" else 0)


def test_tables_are_built_before_the_transform():
    src = code("api.cu")
    body = src[src.index("int invert_impl("):]
    fft = body.index("data_fft<T>(")
    for table in ("ensure_bands(", "fixed_table(", "alpha_tables(", "ensure_wtab(H, o->sources, st));\n    else", "weights_or_null<T>("):
        assert 0 < body.index(table) < fft, table
    multi = code("multi.cu")
    body = multi[multi.index("int invert_multi("):]
    assert body.index("ensure_multi_tables(") < body.index("multi_data(")
