"""Rules of the device code that no run can show broken, checked in its text:
the hardware leaves open what would go wrong, so a kernel that breaks one may
still give the right values on the chip at hand."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_3422_gb300", "csrc")


def code(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"/\*.*?\*/|//[^\n]*", "", text, flags=re.S)


def functions(text):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__\s+void[^;{]*?(\w+)\s*\((?:[^()]|\([^()]*\))*\)\s*\{", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        yield m.group(1), text[m.end():i]


@pytest.mark.parametrize("kernel", ["prop_tile_kernel", "prop_duo_kernel"])
def test_a_commit_comes_from_the_lane_that_issued_the_products(kernel):
    """tcgen05.commit tracks the MMAs of its own thread, and which lane
    elect.sync picks is not specified: a commit of a fixed lane may track none."""
    body = dict(functions(code("ge_prop.cu")))[kernel]
    assert re.search(r"bool leader = elect_one\(\)", body)
    assert re.findall(r"\btc_commit\w*\(\w+", body) == ["tc_commit_if(leader"]


def test_a_tile_buffer_is_fenced_before_tma_writes_it_again():
    """The rounds of a launch use the same two buffers, which threads wrote and
    read before: a proxy fence between those accesses and the copy, at every load."""
    loads = [m.start() for m in re.finditer(r"\btma_load_rows\(", code("ge_tb.cu"))]
    assert len(loads) == 2
    for at in loads:
        before = code("ge_tb.cu")[:at]
        assert re.search(r"fence_proxy_async_smem\(\);\s*mbar_arrive_expect_tx\([^;]*\);\s*$", before)
