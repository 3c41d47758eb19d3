"""Every wait of the kernels is bounded, checked in their sources (a wait that could last for good is not made to happen on a GPU)."""
import glob
import os
import re

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
