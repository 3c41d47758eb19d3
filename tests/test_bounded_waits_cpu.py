"""Every wait of the kernels is bounded, checked in their sources (a wait that could last for good is not made to happen on a GPU)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_21317_b200", "csrc")


def test_no_named_barriers():
    """A warp whose bounded wait runs out leaves for the end of the kernel.  Warps that meet it at a named barrier (bar.sync / barrier.sync with a
    number of threads) would wait there without limit, so warps of a part of the CTA meet at mbarriers, whose waits are bounded."""
    found = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        code = re.sub(r"//.*", "", open(path).read())
        for m in re.finditer(r"\b(bar|barrier)\.(cta\.)?(sync|red|arrive)\b[^\"]*", code):
            found.append((os.path.basename(path), m.group(0)))
    assert not found, found


# (file, where the code of whole warps begins, where it ends): waits there are followed by instructions that take the whole warp
WARP_ROLES = [
    ("httm_attention_tc.cu", "bool epilogue_part(", "attention_tc_kernel("),
    ("httm_attention_tc.cu", "softmax + epilogue", "tmem_dealloc"),
    ("httm_big_blocks.cu", "arg-max over the chunk's dst tokens", "tmem_dealloc"),
    ("httm_linear.cu", "epilogue: lane = row", "tcgen05.dealloc"),
    ("httm_mem_kernels.cu", "int buf = 0;", "if (failed)"),
    ("httm_small_blocks.cu", "int it = 0;", "if (failed) break;"),
]


@pytest.mark.parametrize("name,start,end", WARP_ROLES, ids=["parts", "softmax", "scores", "linear", "deviation", "match_small"])
def test_a_warp_gives_up_as_a_whole(name, start, end):
    """The lanes of a warp poll a barrier each for itself, and one may see the time-out where the next still sees the barrier complete.  The
    loads from tensor memory, votes and shuffles behind the wait need all lanes, so the outcome of every wait is a vote of the warp."""
    code = open(os.path.join(CSRC, name)).read()
    begin = code.index(start)
    code = re.sub(r"//.*", "", code[begin:code.index(end, begin)])
    waits = [m.start() for m in re.finditer(r"mbar_wait\w*\(", code)]
    assert waits
    for at in waits:
        statement = code[max(code.rfind(c, 0, at) for c in ";{}") + 1:at]
        assert "__all_sync(0xffffffffu," in statement, code[at - 60:at + 60]
