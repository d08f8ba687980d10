"""The look at a batch's end votes and shuffles over the whole warp, so whether to look has to be the same on
every lane: what decides it comes from one lane's reading of the timer."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_10158_gb300", "csrc",
                   "exec_common.cuh")


def test_the_decision_to_look_is_one_lanes():
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    body = text[text.index("void group_loop("):]
    assert "__shfl_sync(0xffffffffu, (uint32_t)globaltimer(), 0)" in re.search(
        r"uint32_t look = ([^;]*);", body).group(1)
    later = re.findall(r"\n\s+look = ([^;]*);", body)
    assert later and all(x.startswith("wnow +") for x in later)
    assert re.search(r"wnow = __shfl_sync\(0xffffffffu, \(uint32_t\)t1, 0\)", body)
    assert re.search(r"if \(\(int32_t\)\(wnow - look\) >= 0\)", body)
