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
    ("httm_mem_kernels.cu", "for (int64_t task = first; task < n_tasks; task += stride, cur.advance()", "if (failed)"),
    ("httm_small_blocks.cu", "for (int64_t task = first; task < n_tasks; task += stride)", "if (failed) break;"),
    ("httm_small_blocks.cu", "for (int64_t unit = first; unit < n_units; unit += stride)", "if (failed) break;"),
]


@pytest.mark.parametrize("name,start,end", WARP_ROLES, ids=["parts", "softmax", "scores", "linear", "deviation", "match_small", "merge_small"])
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


@pytest.mark.parametrize("kernel", ["match_team_kernel", "merge_team_kernel"])
def test_a_team_gives_up_as_a_whole(kernel):
    """In the kernels with a team of warps per block a thread only notes that its wait ran out; the team leaves after a vote of all its threads."""
    code = open(os.path.join(CSRC, "httm_mid_blocks.cu")).read()
    begin = code.index("for (int64_t unit = blockIdx.x;", code.index(kernel + "(const __grid_constant__"))
    code = re.sub(r"//.*", "", code[begin:code.index("\n    }\n", begin)])
    waits = [code[code.rfind(";", 0, m.start()) + 1:m.start()].strip() for m in re.finditer(r"mbar_wait\w*\(", code)]
    assert waits == ["const bool arrived ="] and "return" not in code
    leaves = re.findall(r"if \(([^{;]*)\) (?:\{\s*failed = \w+;\s*)?break;", code)
    assert len(leaves) == code.count("break;") and set(leaves) <= {"team_any<W>(!arrived)", "failed", "failed >= 0"}, leaves


@pytest.mark.parametrize("kernel,tensors", [("match_small_kernel", 2), ("merge_small_kernel", 3)])
def test_a_warp_that_gives_up_waits_for_every_load_in_flight(kernel, tensors):
    """The loads of a warp are numbered in the order in which they are issued and awaited.  With two stages the first two are issued ahead and another behind
    every one that has arrived, so all that is in flight when number `seq` does not arrive is that one and, unless it is the last, the next.  Checked
    on the kernel's own expressions."""
    code = open(os.path.join(CSRC, "httm_small_blocks.cu")).read()
    begin = code.index(kernel + "(const __grid_constant__")
    code = re.sub(r"//.*", "", code[begin:code.index("\n}\n", begin)])
    ahead = re.search(r"failed = true;\s*ahead = ([^;]*);", code).group(1).replace("&&", " and ").replace("||", " or ").replace("!", " not ")
    for units in (1, 2, 3):
        for seq in range(tensors * units):
            unit, t = divmod(seq, tensors)
            issued = min(2 + seq, tensors * units)
            assert eval(ahead, {"UNITS": True, "SPLIT": False, "t": t, "more": unit + 1 < units}) == (issued > seq + 1), (unit, t)
    assert not eval(ahead, {"UNITS": False, "SPLIT": True, "t": 0, "more": True})   # (a tensor at a time, through one stage)
    # and it waits for them where and in the phase in which the loop would
    stage = re.search(r"uint32_t st = ([^;]*);", code).group(1)
    waits = [re.sub(r"\bst\b", "(" + stage + ")", w) for w in re.findall(r"mbar_wait_bounded\((.*?), a\.status", code)]
    assert len(waits) == 2 and "i <= seq + (ahead ? 1 : 0)" in code
    assert re.sub(r"\bi\b", "seq", waits[1]) == waits[0], waits
