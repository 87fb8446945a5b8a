"""Every wait of a whole warp must end the same way for all its lanes (mbar_wait_uniform): mbar_wait decides lane by
lane, so it may only stand where a single lane runs."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2309_12307_b200", "csrc")


@pytest.mark.parametrize("name", ["fwd_kernel.cu", "bwd_kernels.cu"])
def test_lanes_wait_alone_only_where_one_lane_runs(name):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    found, single_lane = 0, []  # single_lane: per open brace, whether it opened the body of a one-lane branch
    for m in re.finditer(r"\bif \(lane == 0\) \{|\bif \(elect_one\(\)\) \{|\{|\}|\bmbar_wait\(|\bmbar_wait_drain\(", text):
        token = m.group()
        if token.endswith("{"):
            single_lane.append(token != "{")
        elif token == "}":
            single_lane.pop()
        else:
            found += 1
            assert any(single_lane), f"{name}: {token} of a whole warp in line {text.count(chr(10), 0, m.start()) + 1}"
    assert found > 0 and not single_lane
