"""The bounded waits of the tensor-core kernels, read from their sources (no GPU: a wait that runs out needs a fault).

A wait that may end its loop is one lane's (MMA issue, bulk copies); a whole warp waits by tc::warp_wait and goes on in step
whatever comes.  Where each lane of a warp decided for itself, some could give up while the others went on to
tcgen05.ld.sync.aligned and full-warp barriers.  What a lane has issued, MMAs and bulk copies, has ended before the CTA
frees tensor memory and leaves its shared memory.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1308_2445_gb300", "csrc")
ONE_LANE = ("if (lane == 0)", "if (tid == 0)")


def source(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())


def enclosing_heads(text, pos):
    """The text in front of every brace that is open at pos."""
    heads, depth = [], 0
    for i in range(pos - 1, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            if depth == 0:
                start = max(text.rfind(c, 0, i) for c in ";{}")
                heads.append(text[start + 1:i].strip())
            else:
                depth -= 1
    return heads


@pytest.mark.parametrize("name", ["gram_tc.cu", "update_tc.cu", "oz.cu"])
def test_waits_are_one_lane_s_or_a_whole_warp_s(name):
    text = source(name)
    heads = [enclosing_heads(text, m.start()) for m in re.finditer(r"tc::mbar_wait\(", text)]
    heads = [h for h in heads if any("__global__" in x for x in h)]   # a kernel's own waits
    assert heads and "tc::warp_wait(" in text
    assert all(any(x.endswith(ONE_LANE) for x in h) for h in heads)
    # nothing hangs on a warp's wait
    assert all(text[:m.start()].rstrip().endswith((";", "{", "}", ")")) for m in re.finditer(r"tc::warp_wait\(", text))


@pytest.mark.parametrize("name", ["gram_tc.cu", "update_tc.cu", "oz.cu"])
def test_issued_work_ends_before_the_cta(name):
    text = source(name)
    issuers = len(re.findall(r"tc::mma_commit\(&(?:done|phasedone|segdone)\)", text))
    assert issuers and len(re.findall(r"tc::mma_drain\(&drain", text)) == issuers
    assert len(re.findall(r"bulk_copy\(base", text)) == len(re.findall(r"drain_copies\(wfull", text))
