"""Rules of the kernels' mbarrier protocols whose breach could only show as a hang, checked without a GPU.

A wait asks for a phase by its parity, so it is sound only while its thread is never two phases behind the barrier."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_12471_b200", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


# An issuing warp: all lanes wait, one issues, and only what it issues lets the barriers move on.  The other lanes keep up only where a
# vote stands between a wait and the next thing issued.
@pytest.mark.parametrize("name,end", [("attn_tc.cu", "softmax, one thread per row"), ("attn_tc32.cu", "converters: fp32 rows")])
def test_waits_of_issuing_warps_end_in_a_vote(name, end):
    text = _source(name)
    start = text.index("leader = elect_one()")
    lines = text[start:text.index(end, start)].splitlines()
    waits = [i for i, line in enumerate(lines) if re.search(r"\bmbar_wait\w*\(", line) and "mbar_wait_drain(" not in line]
    assert len(waits) >= 4
    for i in waits:
        voted = re.search(r"\bmbar_wait4?_warp\(", lines[i]) or any("__all_sync" in line for line in lines[i:i + 4])
        assert voted, lines[i]
        if not re.search(r"\bmbar_wait4?_warp\(", lines[i]):
            until = next(k for k in range(i, i + 4) if "__all_sync" in lines[k])
            assert not any("leader" in line for line in lines[i:until])
