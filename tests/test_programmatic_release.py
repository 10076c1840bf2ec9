"""A kernel that allocates tensor memory releases its programmatic successor only after the block-wide barrier that
follows the allocation.  Released earlier, a successor's block on the same SM could take the columns and hold them while
it waits for this kernel, whose allocation would then wait for it."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_01216_gb300", "csrc")


def kernels():
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        for part in re.split(r"(?=__global__ )", src)[1:]:
            yield name, part


def test_release_follows_the_allocation():
    seen = 0
    for name, body in kernels():
        a, r = body.find("tmem_alloc("), body.find("pdl_release()")
        if a < 0 or r < 0:
            continue
        seen += 1
        assert a < body.find("__syncthreads()", a) < r, (name, body[:80])
    assert seen >= 2
